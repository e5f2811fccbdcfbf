"""Resampling and observables at the sizes where their launches change shape.

* pa_resample_static at the edges of runs (32), weights blocks (1024) and scan
  blocks, with energies that take each way to the weights: a few levels per
  block, more levels than a block looks up, energies not congruent modulo 4, one
  replica that takes nearly every slot, equal energies.  Parents bit-exact
  against the oracle; ln Q to 1e-12 as in test_gpu_parity.
* Populations around the largest that one cluster resamples (8192: also the static
  call), the largest whose weights launch completes the prefix (131072), above it,
  and above 2048 weights blocks (segments of two): one step of a 2D L = 2
  population against the oracle's resampling of the downloaded energies, and
  the observables against integer sums and family counts of the downloads.
  S_f sums at most R terms c ln c of FP64: its relative error is below
  R 2^-53 < 1e-9, and ln R - sum / R is compared to 1e-8 absolute.
"""
import numpy as np
import pytest

from paper_1710_09025_gb300 import workloads as W
from test_gpu_fullsize import _pairs

pytestmark = pytest.mark.gpu


def _energies(how, R, rng):
    if how == "levels":
        return 4 * rng.integers(-150, -90, R)
    if how == "wide":
        return 4 * rng.integers(-3000, 3000, R)
    if how == "odd":
        return rng.integers(-500, -400, R)
    if how == "one":
        E = np.full(R, 400)
        E[R // 3] = -1000
        return E
    return np.full(R, -96)


@pytest.mark.parametrize("R", [1, 2, 31, 32, 33, 1023, 1024, 1025, 2049, 4097, 8191, 8192, 8193, 32769, 65535, 65536])
@pytest.mark.parametrize("how", ["levels", "wide", "odd", "one", "equal"])
def test_static_resample_edges(pa, oracle, R, how):
    import torch
    E = _energies(how, R, np.random.default_rng(R)).astype(np.int32)
    e = torch.from_numpy(E).cuda()
    par = torch.full((R,), -1, dtype=torch.int32, device="cuda")
    lnq = torch.empty(1, dtype=torch.float64, device="cuda")
    pa.pa_resample_static(e.data_ptr(), R, 0.5, 0.52, 9, 4242 + R, 3, 2, par.data_ptr(), lnq.data_ptr())
    torch.cuda.synchronize()
    want = oracle.resample(0, _pairs(E, 0), 0.5, 0.52, 9, 4242 + R, 3, 2)
    np.testing.assert_array_equal(par.cpu().numpy(), want["parent"])
    assert lnq.item() == pytest.approx(want["lnQ"], rel=1e-12, abs=1e-13)


@pytest.mark.parametrize("R", [1025, 8192, 8193, 131071, 131072, 131073, 400_001, 2_098_177])
def test_population_resample_sizes(pa, oracle, R):
    P, O = pa, oracle
    J, betas, seed = W.couplings_pm(2, 2, 5), np.array([0.0, 0.4, 1.1]), 99 + R
    pop = P.Population(2, 2, P.PA_PM1, J, None, R, betas, 1, seed)
    try:
        assert pop.step()
        fam = P.pa_get_family(pop.ctx)
        for k in (1, 2):
            want = O.resample(0, _pairs(P.pa_get_energies(pop.ctx, 0), 0), betas[k - 1], betas[k], k, seed)
            assert pop.step()
            par = P.pa_get_parents(pop.ctx)
            np.testing.assert_array_equal(par, want["parent"])
            fam = fam[par]
            np.testing.assert_array_equal(P.pa_get_family(pop.ctx), fam)
            E = P.pa_get_energies(pop.ctx, 0)
            o = pop.observables(k)
            assert o["E_mean"] == int(E.sum()) / R and o["E2_mean"] == int((E * E).sum()) / R
            assert o["lnQ"] == pytest.approx(want["lnQ"], rel=1e-12, abs=1e-13)
            c = np.unique(fam, return_counts=True)[1].astype(np.float64)
            assert o["S_f"] == pytest.approx(np.log(R) - (c * np.log(c)).sum() / R, abs=1e-8)
    finally:
        pop.close()


@pytest.mark.parametrize("R,beta", [(5000, 3.0), (131073, 2.5)])
def test_long_families(pa, oracle, R, beta):
    """Runs of one family over many 1024-replica windows of the observables:
    one large temperature step leaves few ancestors."""
    P = pa
    J, betas, seed = W.couplings_pm(3, 4, 8), np.array([0.0, beta, beta + 0.1]), 7
    pop = P.Population(3, 4, P.PA_PM1, J, None, R, betas, 1, seed)
    try:
        for k in range(3):
            assert pop.step()
        fam = P.pa_get_family(pop.ctx)
        c = np.unique(fam, return_counts=True)[1].astype(np.float64)
        assert c.max() > 300
        assert pop.observables(2)["S_f"] == pytest.approx(np.log(R) - (c * np.log(c)).sum() / R, abs=1e-8)
    finally:
        pop.close()


@pytest.mark.parametrize("R", [33, 1000, 8193, 33_025, 131_072, 131_073])
def test_real_population_resample_sizes(pa, oracle, R):
    """Real couplings: 256-replica weights blocks up to 131072 replicas
    (ln Q as test_gpu_fullsize compares it)."""
    P, O = pa, oracle
    J, betas, seed = W.couplings_gauss(2, 2, 5), np.array([0.0, 0.4, 2.1]), 7 + R
    pop = P.Population(2, 2, P.PA_REAL, J, None, R, betas, 1, seed)
    try:
        assert pop.step()
        for k in (1, 2):
            want = O.resample(1, _pairs(P.pa_get_energies(pop.ctx, 1), 1), betas[k - 1], betas[k], k, seed)
            assert pop.step()
            np.testing.assert_array_equal(P.pa_get_parents(pop.ctx), want["parent"])
            assert pop.observables(k)["lnQ"] == pytest.approx(want["lnQ"], rel=1e-10, abs=1e-10)
    finally:
        pop.close()
