"""Tabu search where one warp owns every variable, on both sides of its limits
(4 and 8 variables per thread), with the compact and the wide keys."""
import pytest

from tests.test_gpu_parity import L, Problem, _check_tabu, _tabu_both_keys, random_solutions  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("asp", [0, 1])
@pytest.mark.parametrize("n,variant", [(1, -1), (3, -1), (127, -1), (128, -1), (129, -1), (255, -1), (256, -1), (257, -1),
                                       (128, 1), (256, 0)])
def test_search_equals_oracle(L, orc, n, variant, asp):  # noqa: F811
    R, alpha, c = 2, 4 * n + 1, max(1, n // 9)
    P = Problem(n, 0.8, 3 * n + 1, R=R)
    X0 = random_solutions(n, R, n + 5)
    for res in _tabu_both_keys(P, X0, alpha, c, asp, variant):
        _check_tabu(orc, P.Q, X0, alpha, c, asp, res)
    P.close()


@pytest.mark.parametrize("n", [1024, 1025, 2560, 2561])
def test_blocks_of_several_warps_equal_oracle(L, orc, n):  # noqa: F811
    """Both sides of 20 warps, up to which every thread keeps the objective."""
    R, alpha, c = 2, 400, n // 50
    P = Problem(n, 0.3, n + 1, R=R)
    X0 = random_solutions(n, R, n + 6)
    for res in _tabu_both_keys(P, X0, alpha, c, 0, -1):
        _check_tabu(orc, P.Q, X0, alpha, c, 0, res)
    P.close()
