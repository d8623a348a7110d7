"""The selection's radix sort at the sizes where it can go wrong (warp runs of
32, the largest n) and with keys that agree in most bits, in none or in all."""
import numpy as np
import pytest

from paper_2502_13947_gb300 import icd2s as I
from paper_2502_13947_gb300.instances import make_qubo
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,K,m,w", [(31, 3, 9, (65536, 65536, 32768)), (1023, 64, 15, (65536, 65536, 32768)),
                                     (1025, 5, 200, (0, 0, 0)), (4097, 16, 256, (1 << 24, -(1 << 24), 1 << 24)),
                                     (16384, 64, 256, (1 << 24, 1 << 24, -(1 << 24)))])
def test_groups_are_the_highest_ranked(n, K, m, w):
    torch = torch_cuda()
    q = I.icd2s_qubo_create(make_qubo(n, 0.2, 3))
    R = 3
    st = I.icd2s_state_create(q, R, 9)
    I.icd2s_tabu(st, min(n, 400), max(2, n // 150))
    idx = torch.full((R * K * m + 1,), -1, dtype=torch.int32, device="cuda")
    off = torch.zeros(R * K + 1, dtype=torch.int32, device="cuda")
    sp = I.SelectParams(w1=w[0], w2=w[1], w3=w[2], K=K, m_min=max(1, m // 2), m_max=m, iter=4)
    I.icd2s_select_subqubos(st, sp, idx.data_ptr(), off.data_ptr())
    A, _, _ = I.icd2s_get_control(st, R, n)
    idx, off = idx.cpu().numpy(), off.cpu().numpy()
    for p in range(R):
        rank = np.lexsort((np.arange(n), -A[p].astype(np.int64)))   # A descending, index ascending
        o = off[p * K:(p + 1) * K + 1]
        for k in range(K):
            want = np.sort(rank[o[k] - o[0]:o[k + 1] - o[0]])
            assert np.array_equal(idx[o[k]:o[k + 1]], want), (p, k)
    I.icd2s_state_destroy(st)
    I.icd2s_qubo_destroy(q)
