"""Recomputed gains and energies on both sides of the lines between their paths: dp4a or
tensor cores by n and the number of solutions, one or several CTAs per row beyond."""
import numpy as np
import pytest

from paper_2502_13947_gb300 import icd2s as I
from paper_2502_13947_gb300.instances import make_qubo, random_solutions

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,R", [(513, 65), (1023, 448), (1023, 449), (1100, 321), (1025, 383), (1025, 385), (2499, 1),
                                 (2500, 1), (8192, 2), (8193, 2)])
def test_loaded_solutions_have_the_exact_gains(n, R):
    Q = make_qubo(n, 1.0, n, lo=-128, hi=127)
    X = random_solutions(n, R, 3)
    X[0] = 1
    Qf, Xf = Q.astype(np.float32), X.astype(np.float32)   # sums below 2^24: exact in float
    H = (Xf @ Qf).astype(np.int64)
    d, Xi = np.diag(Q).astype(np.int64), X.astype(np.int64)
    q = I.icd2s_qubo_create(Q)
    st = I.icd2s_state_create(q, R, 5)
    for _ in range(2):
        I.icd2s_state_load(st, X)
        x, g, e = I.icd2s_get_state(st, R, n)
        assert np.array_equal(x, X) and np.array_equal(e, (H * Xi).sum(1))
        assert np.array_equal(g, (1 - 2 * Xi) * (d + 2 * (H - Xi * d)))
    I.icd2s_state_destroy(st)
    I.icd2s_qubo_destroy(q)
