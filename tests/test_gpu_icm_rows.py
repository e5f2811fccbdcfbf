"""Cluster moves grow islands by x-rows of L bits: the row widths and counts
where that can go wrong, every step bit for bit against the oracle.  Rows of
less than a word that start inside one (L = 2, 6, 10, 12, 14), rows of a half
and a whole word (16, 32), rows of 64 bits, up to eight rows per lane (3D
L = 16), replicas that fill a group, leave one over, or a single pair, int8 rows
with a partial last vector, and real couplings."""
import numpy as np
import pytest

from paper_1710_09025_gb300 import workloads as W
from test_gpu_icm import _run

pytestmark = pytest.mark.gpu

PM1, REAL = 0, 1


@pytest.mark.parametrize("D,L,R,ns,layout,kind", [
    (2, 2, 65, 2, 0, PM1), (3, 2, 33, 2, 2, PM1), (2, 10, 64, 2, 0, PM1), (2, 12, 130, 2, 2, PM1), (3, 6, 129, 2, 0, PM1),
    (3, 6, 35, 2, 2, PM1), (3, 10, 66, 2, 0, PM1), (3, 12, 31, 2, 0, PM1), (3, 14, 20, 2, 0, PM1), (3, 16, 24, 2, 0, PM1),
    (2, 64, 18, 2, 0, PM1), (2, 64, 9, 2, 2, PM1), (2, 32, 2, 2, 0, PM1), (3, 4, 3, 2, 0, PM1), (3, 4, 1, 2, 0, PM1),
    (2, 16, 5000, 2, 0, PM1), (3, 10, 40, 2, 0, REAL), (2, 32, 50, 2, 0, REAL),
])
def test_icm_rows(pa, oracle, D, L, R, ns, layout, kind):
    J = W.couplings_pm(D, L, 700 + L + D) if kind == PM1 else W.couplings_gauss(D, L, 700 + L + D)
    _run(pa, oracle, D, L, kind, J, R, W.schedule_lb(4, 1.2), ns, 2700 + L, layout=layout)
