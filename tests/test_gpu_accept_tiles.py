"""The guard band of the real-coupling Metropolis decision on the lattices whose
sweeps still use it: 3D L = 12, and 3D L = 10 with a field, have no threshold
table and decide most attempts from the estimate of exp(-x).  With exact_accept = 1
every uphill attempt takes the specified rule; both give the same run bit for bit
over a schedule to beta = 5 (10^9 decisions each, about 10^5 of them inside the
band of relative width 2^-14)."""
import numpy as np
import pytest

from paper_1710_09025_gb300 import workloads as W
from test_gpu_batch import PM1, REAL, _snapshot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,field,R,opts", [(12, False, 1450, {}), (12, True, 1463, {}), (10, True, 2503, {}),
                                            (10, True, 611, dict(threads=128))])
def test_specified_rule_in_every_lane_of_a_tile_gives_the_same_run(pa, L, field, R, opts):
    J = W.couplings_gauss(3, L, 31 + L)
    h = W.field_uniform(L ** 3, 41 + L) if field else None
    betas = W.schedule_lb(41, 5.0)
    runs = []
    for exact in (0, 1):
        pop = pa.Population(3, L, pa.PA_REAL, J, h, R, betas, 10, 99, accumulate_grad=1, exact_accept=exact, **opts)
        pop.run()
        runs.append((pa.pa_get_spins(pop.ctx), pa.pa_get_energies(pop.ctx, pa.PA_REAL), pa.pa_free_energy(pop.ctx))
                    + tuple(pa.pa_get_grad_counts(pop.ctx)))
        pop.close()
    for a, b in zip(*runs):
        np.testing.assert_array_equal(a, b)


def test_batch_tiles_with_the_specified_rule_match(pa):
    """The same in a batch: the tiles run in the mixed launch, beside tables."""
    lattices = [(REAL, 10, True), (REAL, 12, False), (REAL, 12, True), (REAL, 10, False), (PM1, 6, False)]
    insts = [dict(L=L, kind=kind, J=W.instance(3, L, kind, 700 + i)[0], R=200 + 7 * i, rng_instance=i,
                  h=W.field_uniform(L ** 3, 800 + i) if field else None)
             for i, (kind, L, field) in enumerate(lattices)]
    betas = W.schedule_lb(21, 5.0)
    snaps = []
    for exact in (0, 1):
        b = pa.pa_batch_create(3, insts, betas, 10, 4242, pa.pa_options_default(exact_accept=exact))
        try:
            pa.pa_batch_run(b, -1)
            snaps.append([_snapshot(pa, pa.pa_batch_instance(b, i), inst["kind"], len(betas) - 1)
                          for i, inst in enumerate(insts)])
        finally:
            pa.pa_batch_destroy(b)
    for got, want in zip(*snaps):
        for g, w in zip(got[:5], want[:5]):
            np.testing.assert_array_equal(g, w)
        assert got[5] == want[5]


@pytest.mark.parametrize("L,field,R,threads", [(12, True, 333, 0), (12, False, 97, 128), (10, True, 250, 0)])
def test_tiles_match_the_oracle(pa, oracle, L, field, R, threads):
    """Several tiles of 32 replicas and a ragged last one: what the sweeps produce
    (spins, int128 energies, gradient counts) and the parents that follow from it,
    bit for bit."""
    P = pa
    J = W.couplings_gauss(3, L, 61 + L)
    h = W.field_uniform(L ** 3, 62 + L) if field else None
    betas = W.schedule_lb(4, 4.0)
    ref = oracle.Sim(3, L, REAL, J, h, R, betas, 2, 63 + L, accumulate_grad=True)
    pop = P.Population(3, L, REAL, J, h, R, betas, 2, 63 + L, accumulate_grad=1, threads=threads)
    try:
        for k in range(len(betas)):
            assert pop.step()
            ref.step()
            np.testing.assert_array_equal(P.pa_get_spins(pop.ctx), ref.spins(), err_msg=f"spins k={k}")
            np.testing.assert_array_equal(P.pa_get_energies(pop.ctx, REAL), ref.energies_raw(), err_msg=f"E k={k}")
            if k > 0:
                np.testing.assert_array_equal(P.pa_get_parents(pop.ctx), ref.parents(), err_msg=f"parents k={k}")
        for got, want in zip(P.pa_get_grad_counts(pop.ctx), ref.grad_counts()):
            np.testing.assert_array_equal(got, want)
    finally:
        pop.close()
