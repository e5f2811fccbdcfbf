"""Resampling with a population that changes, on each route of the launches: one
cluster (at most 8192 source replicas), a weights launch that completes the prefix
(at most 131072), a run table of its own (above), and for nearest-integer
resampling grids sized for a capacity above each of these limits while the drawn
population lies below it, or beyond the capacity.

2D L = 2, so that the oracle follows populations of 10^5: spins, energies, parents,
families and populations bit for bit.  ln Q and beta F to 1e-12 (+-J) or 1e-10 as
in test_gpu_parity (the sums behind them have one fixed order).  S_f and <E> differ
by the order of at most R FP64 terms: relative 2 R 2^-53 < 1e-10 of sums of which the mean
is at most ln R < 12, or |E| <= 40."""
import numpy as np
import pytest

from paper_1710_09025_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PM1, REAL = 0, 1
GROW = [9000, 20_000, 8192, 140_000, 131_072, 131_073, 5000, 9001, 1]
# capacity, targets
NEAREST = {
    "runs": (150_000, [140_000, 131_072, 131_000, 60_000, 8000, 300, 9000, 140_000]),
    "fused": (100_000, [99_000, 8193, 8000, 33, 20_000, 98_000]),
    "drops": (10_000, [9000, 9995, 9999, 8192, 100, 9998, 9999]),
    "cluster": (8192, [8000, 8190, 3000, 1025, 1024, 8192, 8192, 8192]),
}


def _follow(pa, oracle, kind, R, pops, scheme, capacity=0, layout=0):
    P = pa
    J = W.couplings_pm(2, 2, 5) if kind == PM1 else W.couplings_gauss(2, 2, 6)
    betas = np.linspace(0.0, 0.9, len(pops))
    seed = 71 + len(pops)
    ref = oracle.Sim(2, 2, kind, J, None, R, betas, 1, seed, populations=pops, resampling=scheme, capacity=capacity)
    pop = P.Population(2, 2, kind, J, None, R, betas, 1, seed, populations=pops, resampling=scheme, capacity=capacity,
                       layout=layout)
    tol = 1e-12 if kind == PM1 else 1e-10
    sizes = []
    try:
        for k in range(len(pops)):
            assert pop.step()
            ref.step()
            sizes.append(P.pa_sizes(pop.ctx)["R"])
            assert sizes[-1] == ref.R_now
            np.testing.assert_array_equal(P.pa_get_spins(pop.ctx), ref.spins(), err_msg=f"spins k={k}")
            want = np.array(ref.energies(), np.int64) if kind == PM1 else ref.energies_raw()
            np.testing.assert_array_equal(P.pa_get_energies(pop.ctx, kind), want, err_msg=f"E k={k}")
            if k > 0:
                np.testing.assert_array_equal(P.pa_get_parents(pop.ctx), ref.parents(), err_msg=f"parents k={k}")
            np.testing.assert_array_equal(P.pa_get_family(pop.ctx), ref.family(), err_msg=f"family k={k}")
            o, r = pop.observables(k), ref.obs(k)
            assert o["R"] == r["R"] == sizes[-1]
            assert o["lnQ"] == pytest.approx(r["lnQ"], rel=tol, abs=1e-13)
            assert o["betaF"] == pytest.approx(r["betaF"], rel=tol)
            assert o["S_f"] == pytest.approx(r["S_f"], abs=12e-10)
            assert o["E_mean"] == pytest.approx(r["E_mean"], abs=40e-10)
    finally:
        pop.close()
    return sizes


@pytest.mark.parametrize("kind,layout", [(PM1, 0), (PM1, 2), (REAL, 0)])
def test_multinomial_populations_between_the_routes(pa, oracle, kind, layout):
    assert _follow(pa, oracle, kind, max(GROW), GROW, 0, layout=layout) == GROW


@pytest.mark.parametrize("kind,layout", [(PM1, 0), (PM1, 2), (REAL, 0)])
@pytest.mark.parametrize("route", sorted(NEAREST))
def test_nearest_populations_on_each_route(pa, oracle, route, kind, layout):
    capacity, targets = NEAREST[route]
    sizes = _follow(pa, oracle, kind, targets[0], targets, 1, capacity=capacity, layout=layout)
    assert max(sizes) <= capacity
    if route in ("drops", "cluster"):
        assert capacity in sizes  # copies were dropped
