"""Packed sweeps on either side of the rules that choose their shape on a GPU of
152 SMs: a team of threads per word (few threads to an SM; populations of a few
thousand, as in most other tests, take it), groups spread evenly over the SMs
(less than a wave of full blocks; with late compaction only if they would be
less than four fifths full), full blocks.  Ragged last groups, lattices whose
last 32-site chunk of the gather is partial, and temperatures of every
comparison mode.  Spins, energies and parents bit-exact against the oracle."""
import numpy as np
import pytest

from paper_1710_09025_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,L,R,layout", [
    (3, 4, 64 * 2424 - 5, 1), (3, 4, 64 * 2425 + 1, 1), (3, 4, 64 * 607 + 9, 2), (3, 4, 64 * 609 - 1, 1),
    (3, 4, 64 * 608, 1), (3, 6, 64 * 152 - 3, 1), (3, 6, 64 * 153, 1), (3, 8, 64 * 152, 2), (3, 8, 64 * 153 - 1, 1),
    (3, 4, 64 * 4864 - 7, 1), (3, 4, 64 * 4865, 1), (3, 8, 64 * 972, 1), (3, 8, 64 * 973 - 2, 1),
    (2, 2, 64 * 700 + 3, 1), (3, 6, 64 * 609 + 33, 1), (2, 6, 64 * 610 + 1, 1), (2, 10, 64 * 20 + 7, 1),
])
def test_packed_spread(pa, oracle, D, L, R, layout):
    P = pa
    J, betas = W.couplings_pm(D, L, 300 + L), np.array([0.0, 0.5, 1.3, 3.2, 4.8])
    ref = oracle.Sim(D, L, 0, J, None, R, betas, 1, 71)
    pop = P.Population(D, L, 0, J, None, R, betas, 1, 71, layout=layout)
    try:
        for k in range(len(betas)):
            assert pop.step()
            ref.step()
            np.testing.assert_array_equal(P.pa_get_spins(pop.ctx), ref.spins(), err_msg=f"spins k={k}")
            np.testing.assert_array_equal(P.pa_get_energies(pop.ctx, 0), np.array(ref.energies(), np.int64))
            if k > 0:
                np.testing.assert_array_equal(P.pa_get_parents(pop.ctx), ref.parents())
    finally:
        pop.close()
