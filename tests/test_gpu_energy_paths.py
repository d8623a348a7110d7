"""Energies and recomputed gains at the edges of their paths: one launch up to
n = 512, the tensor cores beyond (tiles of 128 rows of Q and 128 or 256
solutions, ragged in both directions)."""
import numpy as np
import pytest

from paper_2502_13947_gb300 import icd2s as I
from paper_2502_13947_gb300.instances import make_qubo, random_solutions
from tests.gpu_util import dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,rows", [(1, 3), (33, 1), (511, 5), (512, 9), (513, 1), (640, 127), (700, 129), (1153, 257)])
def test_energies_and_gains(n, rows):
    torch = torch_cuda()
    Q = make_qubo(n, 1.0, n, lo=-128, hi=127)
    X = random_solutions(n, rows, 3)
    X[0] = 1
    q = I.icd2s_qubo_create(Q)
    Qf, Xf = Q.astype(np.float64), X.astype(np.float64)
    H = Xf @ Qf
    E = (H * Xf).sum(1).astype(np.int64)
    x_d, E_d = dev(X), torch.empty(rows, dtype=torch.int64, device="cuda")
    for _ in range(2):   # the second call finds the first one's scratch
        E_d.fill_(7)
        I.icd2s_energy(q, x_d.data_ptr(), rows, E_d.data_ptr())
        assert np.array_equal(E_d.cpu().numpy(), E)
    st = I.icd2s_state_create(q, rows, 5)
    I.icd2s_state_load(st, X)
    x, g, e = I.icd2s_get_state(st, rows, n)
    d = np.diag(Qf)
    want = ((1 - 2 * Xf) * (d + 2 * (H - Xf * d))).astype(np.int64)
    assert np.array_equal(x, X) and np.array_equal(g, want) and np.array_equal(e, E)
    I.icd2s_state_destroy(st)
    I.icd2s_qubo_destroy(q)
