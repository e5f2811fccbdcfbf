"""The library's host code against a CUDA runtime without a device
(shims/fake_cudart.cpp): the library's own objects, linked against a runtime that
records calls, keeps each kernel's shared-memory limit per device and refuses
the launches above it, and fails the call that a test names.  Kernels do not
run; what they compute is covered on the GPU."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
STREAM = 0x4000  # a handle that the fake runtime takes for a stream


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    from paper_1710_09025_gb300 import build as B
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    B.build()
    objs = [os.path.join(B.BUILD, s.replace(".cu", ".o")) for s in B.SOURCES]
    out = tmp_path_factory.mktemp("fake") / "libpamc_fake.so"
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-Wl,-Bsymbolic",
                    "-I" + os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include"),
                    os.path.join(ROOT, "tests", "shims", "fake_cudart.cpp"), *objs, "-o", str(out)], check=True)
    return str(out)


class Fake:
    def __init__(self, lib):
        lib.fake_log.restype = ctypes.c_char_p
        lib.fake_fail.argtypes = [ctypes.c_char_p, ctypes.c_int]
        self.lib = lib

    def reset(self):
        self.lib.fake_reset()
        self.lib.fake_device(0)

    def device(self, d):
        self.lib.fake_device(d)

    def fail(self, name, after=0):
        self.lib.fake_fail(name.encode(), after)

    def log(self):
        return self.lib.fake_log().decode().splitlines()

    def launched(self, kernel):
        return [x for x in self.log() if x.startswith("launch ") and kernel in x]


@pytest.fixture
def fake(fake_lib, monkeypatch):
    """(the package bound to the library on the fake runtime, its controls)"""
    import paper_1710_09025_gb300 as P
    monkeypatch.setattr(P, "_lib", None)
    f = Fake(P.load(fake_lib))
    f.reset()
    yield P, f
    f.reset()


def _couplings(kind, L, seed=1):
    from paper_1710_09025_gb300 import workloads as W
    return W.couplings_gauss(3, L, seed) if kind else W.couplings_pm(3, L, seed)


def _batch(P, insts, n=4, sweeps=2, **opts):
    """insts: (kind, L, R, with a field)"""
    from paper_1710_09025_gb300 import workloads as W
    descs = [dict(L=L, kind=kind, J=_couplings(kind, L, i), h=W.field_uniform(L ** 3, i) if field else None, R=R,
                  rng_instance=i) for i, (kind, L, R, field) in enumerate(insts)]
    return P.pa_batch_create(3, descs, np.linspace(0.0, 1.0, n), sweeps, 7, P.pa_options_default(**opts), STREAM)


@pytest.mark.parametrize("first,second", [
    ([(1, 10, 200, False)], [(1, 4, 200, False)]),                            # table launch: about 200 KB, then 70
    ([(0, 16, 200, False)], [(1, 4, 200, False)]),                            # mixed launch: no such item in the second
    ([(1, 12, 200, False), (1, 10, 200, False)], [(0, 4, 200, False), (1, 6, 200, True)]),
    ([(0, 16, 200, False)], [(0, 4, 200, False)]),
])
@pytest.mark.parametrize("tune", [0, -1])
def test_a_batch_leaves_another_batchs_launches_alone(fake, first, second, tune):
    P, f = fake
    a = _batch(P, first, threads=tune)
    b = _batch(P, second, threads=tune)
    try:
        for x in (a, b):
            P.pa_batch_run(x, 2)
            assert P.pa_batch_step(x) and P.pa_batch_step(x)
            assert P.pa_batch_current_step(x) == 4
    finally:
        P.pa_batch_destroy(a)
        P.pa_batch_destroy(b)


@pytest.mark.parametrize("kind,L,field,opts", [
    (0, 16, False, {}), (0, 16, False, dict(layout=2)), (0, 16, False, dict(groups_per_block=2)), (0, 10, False, {}),
    (1, 12, False, {}), (1, 12, True, dict(accumulate_grad=1)), (1, 10, True, dict(threads=128)), (1, 10, False, {}),
    (1, 8, True, {}),
])
def test_every_device_gets_the_shared_memory_limit(fake, kind, L, field, opts):
    """Tiles above 48 KB: the limit is asked for on each device that launches them."""
    from paper_1710_09025_gb300 import workloads as W
    P, f = fake
    for dev in (0, 1, 2, 0):
        f.device(dev)
        h = W.field_uniform(L ** 3, 3) if field else None
        ctx = P.pa_create(3, L, kind, _couplings(kind, L), h, 9000, [0.0, 0.5], 1, 5, P.pa_options_default(**opts), STREAM)
        try:
            assert P.pa_anneal_step(ctx) and P.pa_anneal_step(ctx)
        finally:
            P.pa_destroy(ctx)


def _kernels(log):
    return [x for x in log if x.startswith("launch ")]


@pytest.mark.parametrize("call,after", [("cudaStreamBeginCapture", 0), ("cudaStreamEndCapture", 0),
                                        ("cudaGraphInstantiate", 0), ("cudaGraphLaunch", 0), ("observe_kernel", 40)])
@pytest.mark.parametrize("n", [-1, 50])
def test_an_anneal_makes_its_steps_without_a_graph(fake, call, after, n):
    """pa_anneal enqueues its first steps before it captures the others.  When the
    graph cannot be had it still makes exactly the steps it was asked for, each
    once and in order, and can be called again."""
    P, f = fake
    args = (3, 4, 0, _couplings(0, 4), None, 10_000, np.linspace(0.0, 1.0, 61), 10, 5)
    want = P.pa_create(*args, stream=STREAM)
    got = P.pa_create(*args, stream=STREAM)
    try:
        f.reset()
        for _ in range(61):
            assert P.pa_anneal_step(want)
        steps = _kernels(f.log())
        f.reset()
        f.fail(call, after)
        P.pa_anneal(got, n)
        assert P.pa_current_step(got) == (61 if n < 0 else n)
        if n > 0:
            P.pa_anneal(got, 61 - n)
        assert _kernels(f.log()) == steps
    finally:
        P.pa_destroy(want)
        P.pa_destroy(got)


@pytest.mark.parametrize("call,after", [("cudaStreamBeginCapture", 0), ("cudaGraphInstantiate", 0),
                                        ("cudaGraphLaunch", 0), ("observe_kernel", 3)])
def test_an_anneal_without_eager_steps_is_all_or_nothing(fake, call, after):
    """On the legacy stream nothing runs before the graph: an error leaves the
    context where it was."""
    P, f = fake
    ctx = P.pa_create(3, 4, 0, _couplings(0, 4), None, 10_000, np.linspace(0.0, 1.0, 9), 10, 5, stream=1)
    try:
        f.reset()
        f.fail(call, after)
        with pytest.raises(P.PAError):
            P.pa_anneal(ctx)
        assert P.pa_current_step(ctx) == 0 and not _kernels(f.log())
        P.pa_anneal(ctx)
        assert P.pa_current_step(ctx) == 9 and len(f.launched("observe_kernel")) == 9
    finally:
        P.pa_destroy(ctx)


@pytest.mark.parametrize("first,second", [
    # +-J beside real couplings with and without a field: per-attempt tiles, or the table launch
    ([(0, 4, 7000, False), (1, 10, 300, True)], [(0, 4, 7000, False), (1, 10, 300, False)]),
    # the same lattices with other populations: other lists of items
    ([(0, 6, 300, False), (0, 8, 300, False)], [(0, 6, 90_000, False), (0, 8, 300, False)]),
])
def test_batches_with_other_items_are_tuned_on_their_own(fake, first, second):
    P, f = fake
    tunings = []
    for insts in (first, second, first):
        b = _batch(P, insts)
        try:
            P.pa_batch_run(b, 1)
            f.reset()
            P.pa_batch_run(b, 1)  # the first step that can be tuned
            tunings.append(len(f.launched("sweep_batch_kernel")) > 1)
            assert (P.pa_batch_sweep_config(b)["tuned_ms"] > 0) == tunings[-1]
        finally:
            P.pa_batch_destroy(b)
    assert tunings == [True, True, False]  # the third takes the first one's shape


def _table_launch(P, f, insts):
    """(chunk, items) of a batch's threshold-table launch"""
    b = _batch(P, insts, threads=-1)
    try:
        assert P.pa_batch_step(b)
        items = np.zeros((f.lib.fake_table_items(None, 0), 2), np.int32)
        f.lib.fake_table_items(items.ctypes.data_as(ctypes.c_void_p), items.size)
        return f.lib.fake_table_chunk(), items
    finally:
        P.pa_batch_destroy(b)


@pytest.mark.parametrize("others", [[(1, 12, 60_000, False)], [(1, 10, 60_000, True)], [(0, 8, 60_000, False)]])
def test_chunks_go_by_the_instances_of_the_table_launch(fake, others):
    P, f = fake
    alone, items = _table_launch(P, f, [(1, 4, 8000, False)])
    assert alone == 16 and len(items) == 125  # 2000 groups
    chunk, beside = _table_launch(P, f, [(1, 4, 8000, False)] + others)
    assert chunk == alone
    np.testing.assert_array_equal(beside, items)


def test_table_items_come_by_cost(fake):
    """The most expensive first: sites times replicas of the chunk."""
    P, f = fake
    insts = [(1, 8, 40, False), (1, 6, 120_000, False), (1, 4, 90_000, True), (1, 10, 12, False)]
    chunk, items = _table_launch(P, f, insts)
    n = [len(items[items[:, 0] == i]) for i in range(len(insts))]
    assert n == [-(-((R + 3) // 4) // chunk) for _, _, R, _ in insts]
    cost = [insts[i][1] ** 3 * insts[i][2] / n[i] for i in items[:, 0]]
    assert cost == sorted(cost, reverse=True)


@pytest.mark.parametrize("graph", [False, True])
def test_an_error_beside_the_table_launch_still_joins_it(fake, graph):
    """What follows on the batch's stream waits for the second stream's launch."""
    P, f = fake
    b = _batch(P, [(0, 4, 300, False), (1, 4, 300, False)], n=5, threads=-1)
    try:
        P.pa_batch_run(b, 2)
        f.reset()
        f.fail("sweep_batch_kernel")
        with pytest.raises(P.PAError):
            P.pa_batch_run(b, -1) if graph else P.pa_batch_step(b)
        assert P.pa_batch_current_step(b) == 2
        if graph:  # nothing of the capture runs
            assert not f.launched("")
        else:
            log = f.log()
            at = next(i for i, x in enumerate(log) if "sweep_batch_table_kernel" in x)
            side = log[at].split(" stream ")[1].split()[0]
            assert side != str(STREAM)
            assert log[at + 1].startswith("record ") and log[at + 1].endswith(" stream " + side)
            event = log[at + 1].split()[1]
            assert log[at + 2] == f"wait {event} stream {STREAM}"
        P.pa_batch_run(b, -1)
        assert P.pa_batch_current_step(b) == 5
    finally:
        P.pa_batch_destroy(b)


@pytest.mark.parametrize("insts,chunk,items", [
    ([(1, 4, 2000, True)] * 8, 32, 128),      # one chunk per SM at most, instead of three or four small ones
    ([(1, 10, 2000, False)] * 8, 32, 128),
    ([(1, 8, 1000, False)] * 32, 64, 128),
    ([(1, 4, 200, True)] * 32, 16, 128),
    ([(1, 10, 2000, False)], 8, 63),          # the smallest already leave no SM a second one
    ([(1, 10, 40_000, False)], 32, 313),      # more than the largest chunks on every SM: two per SM
    ([(1, L, 2000, False) for L in (4, 6, 8, 10)], 8, 252),  # the largest lattice's chunks would be the last
])
def test_a_chunk_per_sm_where_the_queue_is_done_earlier(fake, insts, chunk, items):
    P, f = fake
    got, queue = _table_launch(P, f, insts)
    assert (got, len(queue)) == (chunk, items)
