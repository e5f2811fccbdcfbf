"""Batches that live side by side and differ in the size of their items: each
keeps its launches, whatever another one needs, and gives the results of its
instances' own contexts."""
import numpy as np
import pytest

from paper_1710_09025_gb300 import workloads as W
from test_gpu_batch import PM1, REAL, _snapshot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph,tune", [(False, 0), (True, 0), (True, -1)])
def test_a_batch_of_small_items_beside_one_of_large_ones(pa, graph, tune):
    P = pa
    betas, ns, seed = W.schedule_lb(5, 2.0), 2, 31

    def batch(insts):
        descs = [dict(L=L, kind=kind, J=W.instance(3, L, kind, 50 + i)[0],
                      h=W.field_uniform(L ** 3, i) if field else None, R=R, rng_instance=i)
                 for i, (kind, L, R, field) in enumerate(insts)]
        return descs, P.pa_batch_create(3, descs, betas, ns, seed, P.pa_options_default(threads=tune))

    # the largest item of either launch, then batches without any, or with small ones
    both = [batch([(REAL, 10, 90, False), (PM1, 10, 130, False), (REAL, 12, 40, False), (PM1, 16, 70, False)]),
            batch([(REAL, 4, 100, False)]), batch([(PM1, 4, 100, False), (REAL, 4, 60, True)])]
    try:
        for _, b in both:
            if graph:
                P.pa_batch_run(b, -1)
            else:
                while P.pa_batch_step(b):
                    pass
        k = len(betas) - 1
        for descs, b in both:
            for i, d in enumerate(descs):
                single = P.Population(3, d["L"], d["kind"], d["J"], d["h"], d["R"], betas, ns, seed,
                                      rng_instance=d["rng_instance"])
                single.run(graph=False)
                got = _snapshot(P, P.pa_batch_instance(b, i), d["kind"], k)
                want = _snapshot(P, single.ctx, d["kind"], k)
                for g, w in zip(got[:5], want[:5]):
                    np.testing.assert_array_equal(g, w)
                assert got[5] == want[5]
                single.close()
    finally:
        for _, b in both:
            P.pa_batch_destroy(b)
