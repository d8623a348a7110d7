"""Tabu search on both sides of the block sizes up to which every thread keeps the
objective: 22 warps with the compact keys and the parity labels (16 with signed rows), 8
with the wide keys."""
import pytest

from paper_2502_13947_gb300 import icd2s as I
from paper_2502_13947_gb300.instances import make_qubo
from tests.test_gpu_parity import L, Problem, _check_tabu, _tabu_both_keys, random_solutions  # noqa: F401

pytestmark = pytest.mark.gpu


class Positive(Problem):
    def __init__(self, n, seed, R):
        self.n, self.R = n, R
        self.Q = make_qubo(n, 1.0, seed, lo=0, hi=127)
        self.q = I.icd2s_qubo_create(self.Q)
        self.st = I.icd2s_state_create(self.q, R, 11)


@pytest.mark.parametrize("n", [1024, 1025, 2048, 2049, 2816, 2817])
def test_compact_and_wide_keys_equal_oracle(L, orc, n):  # noqa: F811
    R, alpha, c = 2, 400, n // 50
    P = Problem(n, 0.3, n + 1, R=R)
    X0 = random_solutions(n, R, n + 6)
    for res in _tabu_both_keys(P, X0, alpha, c, 0, -1):
        _check_tabu(orc, P.Q, X0, alpha, c, 0, res)
    P.close()


@pytest.mark.parametrize("n", [2100, 2816, 2817])
def test_parity_labels_equal_oracle(L, orc, n):  # noqa: F811
    """Positive entries: the gain bound lies one bit above the compact keys' on indices."""
    R, alpha, c = 2, 400, n // 50
    P = Positive(n, n + 1, R)
    assert 1 << 18 <= I.icd2s_qubo_gain_bound(P.q) + 1 < 1 << 19
    X0 = random_solutions(n, R, n + 6)
    for res in _tabu_both_keys(P, X0, alpha, c, 0, -1):
        _check_tabu(orc, P.Q, X0, alpha, c, 0, res)
    P.close()
