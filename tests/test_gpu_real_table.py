"""Threshold-table sweeps of real couplings against the oracle, at the sizes
where the tiling can go wrong: one to five replicas (groups of four), planes of
32 and their remainders, fewer replicas than blocks, several chunks per block
(more than 512 replicas a block at L = 2), lattices whose quads do not fill a
warp or have missing sites, tables of whole thresholds (3D L <= 8, 2D) and of
upper halves (3D L = 10, and L = 8 with a field, where about one attempt in
65536 evaluates the rule itself), a field that is zero, one site only, or
everywhere, N_S = 0 and the largest couplings.  What the sweeps produce is
compared bit for bit: spins, int128 energies, gradient counts, and through the
resampling every later step (parents, families)."""
import numpy as np
import pytest

from paper_1710_09025_gb300 import workloads as W

pytestmark = pytest.mark.gpu

REAL = 1


@pytest.mark.parametrize("D,L,R,nt,ns,field,grad", [
    (3, 2, 1, 4, 2, "none", True), (3, 2, 300_001, 3, 1, "uniform", True), (2, 2, 5, 4, 3, "uniform", True),
    (3, 4, 3, 5, 3, "none", False), (3, 4, 1027, 4, 2, "uniform", True), (3, 4, 90_000, 2, 1, "none", True),
    (3, 6, 4, 4, 2, "uniform", True), (3, 6, 5003, 3, 2, "none", True), (3, 8, 33, 4, 2, "none", True),
    (3, 8, 1221, 3, 2, "uniform", True), (3, 10, 2503, 3, 2, "none", True), (3, 10, 31, 3, 2, "uniform", True),
    (3, 12, 21, 3, 1, "uniform", False), (2, 4, 2049, 5, 3, "uniform", True), (2, 6, 131, 5, 2, "none", True),
    (2, 10, 67, 4, 2, "uniform", True), (2, 12, 95, 4, 2, "none", True), (2, 16, 641, 4, 2, "uniform", True),
    (2, 32, 129, 3, 2, "none", True), (2, 32, 30, 3, 1, "uniform", False), (3, 6, 77, 4, 0, "none", True),
    (3, 4, 65, 5, 3, "zero", True), (3, 4, 65, 5, 3, "one", True), (3, 6, 50, 4, 2, "large", True),
])
def test_real_table_parity(pa, oracle, D, L, R, nt, ns, field, grad):
    N = L ** D
    J = W.couplings_gauss(D, L, 4000 + 10 * L + D)
    h = None if field == "none" else W.field_uniform(N, 77 + L)
    if field == "zero":
        h[:] = 0.0
    elif field == "one":
        h[1:] = 0.0
    elif field == "large":
        J, h = np.float32(900.0) * J, np.float32(4000.0) * h
    betas = W.schedule_lb(nt, 2.5)
    P = pa
    ref = oracle.Sim(D, L, REAL, J, h, R, betas, ns, 31 + R, accumulate_grad=grad)
    pop = P.Population(D, L, REAL, J, h, R, betas, ns, 31 + R, accumulate_grad=int(grad))
    try:
        for k in range(nt):
            assert pop.step()
            ref.step()
            np.testing.assert_array_equal(P.pa_get_spins(pop.ctx), ref.spins(), err_msg=f"spins k={k}")
            np.testing.assert_array_equal(P.pa_get_energies(pop.ctx, REAL), ref.energies_raw(), err_msg=f"E k={k}")
            if k > 0:
                np.testing.assert_array_equal(P.pa_get_parents(pop.ctx), ref.parents(), err_msg=f"parents k={k}")
            np.testing.assert_array_equal(P.pa_get_family(pop.ctx), ref.family())
        if grad:
            for got, want in zip(P.pa_get_grad_counts(pop.ctx), ref.grad_counts()):
                np.testing.assert_array_equal(got, want)
    finally:
        pop.close()
