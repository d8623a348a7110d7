"""The exact Ising machine at the edges of its split of the positions (five
tried together, up to eleven walked, up to eight fixed per thread) and with
many equal objectives, where the smallest assignment must win."""
import numpy as np
import pytest

from paper_2502_13947_gb300 import icd2s as I
from paper_2502_13947_gb300.instances import make_qubo, random_solutions, random_subsets
from tests.gpu_util import dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo,hi,density", [(-100, 100, 1.0), (-1, 1, 0.3)])
def test_sizes_at_the_edges_of_the_split(orc, lo, hi, density):
    torch = torch_cuda()
    n, sizes = 120, [2, 7, 12, 13, 14, 15, 16, 17]
    Q = make_qubo(n, density, 5, lo=lo, hi=hi)
    q = I.icd2s_qubo_create(Q)
    st = I.icd2s_state_create(q, 1, 1)
    X0 = random_solutions(n, 1, 4)
    I.icd2s_state_load(st, X0)
    S = random_subsets(n, sizes, 6)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    idx_d, off_d = dev(S), dev(off)
    mask = torch.zeros((1, n), dtype=torch.uint8, device="cuda")
    dE = torch.zeros(len(sizes), dtype=torch.int64, device="cuda")
    I.icd2s_exact_subqubos_batch(st, idx_d.data_ptr(), off_d.data_ptr(), len(sizes), len(sizes), mask.data_ptr(),
                                 dE.data_ptr())
    mask, dE = mask.cpu().numpy()[0], dE.cpu().numpy()
    for k, m in enumerate(sizes):
        s = S[off[k]:off[k + 1]]
        Qs, _ = orc.subqubo(Q, X0[0], s)
        y, want = orc.exact_subqubo(Qs, X0[0][s])
        assert dE[k] == want, m
        assert np.array_equal(X0[0][s] ^ mask[s], y), m
    I.icd2s_state_destroy(st)
    I.icd2s_qubo_destroy(q)
