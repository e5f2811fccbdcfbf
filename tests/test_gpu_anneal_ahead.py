"""pa_anneal enqueues its first steps one by one and the others as a graph: any
split of the schedule gives the states of repeated pa_anneal_step bit for bit."""
import numpy as np
import pytest

from paper_1710_09025_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("parts", [[1, -1], [2, 3, -1], [-1], [12, 1]])
def test_anneal_parts_equal_steps(pa, kind, parts):
    import torch
    P = pa
    J = W.couplings_pm(3, 4, 3) if kind == 0 else W.couplings_gauss(3, 4, 3)
    betas, R = np.linspace(0.0, 1.2, 13), 300

    def state(pop):
        return (P.pa_get_spins(pop.ctx), P.pa_get_energies(pop.ctx, kind), P.pa_get_family(pop.ctx),
                P.pa_free_energy(pop.ctx), [pop.observables(k) for k in range(len(betas))])

    a = P.Population(3, 4, kind, J, None, R, betas, 5, 21)
    with torch.cuda.stream(torch.cuda.Stream()):  # graphs need a stream of their own
        b = P.Population(3, 4, kind, J, None, R, betas, 5, 21)
    try:
        while a.step():
            pass
        P.pa_profile(b.ctx, True)
        for n in parts:
            P.pa_anneal(b.ctx, n)
        assert not any(P.pa_phase_times(b.ctx)[1].values())  # phases are those of pa_anneal_step
        sa, sb = state(a), state(b)
        for x, y in zip(sa[:4], sb[:4]):
            np.testing.assert_array_equal(np.asarray(x), np.asarray(y))
        assert sa[4] == sb[4]
    finally:
        a.close()
        b.close()
