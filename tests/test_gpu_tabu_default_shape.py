"""Tabu search with the default kernel shape around n = 129..256, where it depends on
aspiration and signed rows: every default is as fast as the shape of 4 variables per
thread within what repeated timings differ by, and equals the oracle."""
import pytest

from paper_2502_13947_gb300 import icd2s as I
from tests.gpu_util import torch_cuda
from tests.test_gpu_parity import L, Problem, _check_tabu, _tabu_both_keys, random_solutions  # noqa: F401

pytestmark = pytest.mark.gpu


def _ms(torch, f):
    best = float("inf")
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("asp,rows", [(0, 1), (0, 2), (1, 1)])
@pytest.mark.parametrize("n", [129, 200, 256])
def test_default_shape(L, orc, n, asp, rows):  # noqa: F811
    torch = torch_cuda()
    R, alpha, c = 4, 3000, 2
    P = Problem(n, 0.8, 3 * n + 1, R=R)
    X0 = random_solutions(n, R, n + 5)
    for res in _tabu_both_keys(P, X0, 200, c, asp):
        _check_tabu(orc, P.Q, X0, 200, c, asp, res)
    run = I.icd2s_tabu_aspiration if asp else I.icd2s_tabu
    s = torch.cuda.current_stream().cuda_stream
    ms = {}
    for v in (-1, 0):
        I.icd2s_set_tuning(P.st, tabu_variant=v, tabu_rows=rows)
        P.load(X0)
        ms[v] = _ms(torch, lambda: run(P.st, alpha, c, s))
    P.close()
    assert ms[-1] <= 1.12 * ms[0], ms   # the slower default took 1.2 times as long
