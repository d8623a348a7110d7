"""The write-back around the longest list that is not split: 64 flips, 16 in clusters of
one or two CTAs (many solutions); 16- and 4-byte row loads."""
import numpy as np
import pytest

from paper_2502_13947_gb300 import icd2s as I
from paper_2502_13947_gb300.instances import make_qubo, random_solutions
from tests.gpu_util import dev, torch_cuda
from tests.test_gpu_apply_splits import _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,R,ld", [(2500, 6, 2500), (300, 200, 304), (300, 500, 300), (300, 700, 304), (2100, 12, 2112)])
def test_lists_around_the_limit(n, R, ld):
    torch = torch_cuda()
    Q = make_qubo(n, 1.0, 3, lo=-128, hi=127)
    X = random_solutions(n, R, 4)
    rng = np.random.default_rng(1)
    M = np.zeros((R, n), np.uint8)
    for p in range(R):
        M[p, rng.permutation(n)[:(1, 15, 16, 17, 64, 65)[p % 6]]] = 1
    g, E = _state(Q, X)
    want_g, want_E = _state(Q, X ^ M)
    q = I.icd2s_qubo_create(Q)
    st = I.icd2s_state_create(q, R, 1)
    I.icd2s_state_load(st, X)
    M_d = dev(M)
    for _ in range(2):   # there and back
        I.icd2s_apply_flips_update_gains(st, M_d.data_ptr())
        x1, g1, e1 = I.icd2s_get_state(st, R, n)
        if _ == 0:
            assert np.array_equal(x1, X ^ M) and np.array_equal(g1, want_g) and np.array_equal(e1, want_E)
    assert np.array_equal(x1, X) and np.array_equal(g1, g) and np.array_equal(e1, E)
    I.icd2s_state_destroy(st)
    I.icd2s_qubo_destroy(q)
    Qp, Xp, gp = np.zeros((n, ld), np.int8), np.full((R, ld), 7, np.uint8), np.full((R, ld), -5, np.int32)
    Qp[:, :n], Xp[:, :n], gp[:, :n] = Q, X, g
    Q_d, X_d, g_d, E_d = dev(Qp), dev(Xp), dev(gp), dev(E)
    I.icd2s_apply_flips_static(Q_d.data_ptr(), n, ld, R, M_d.data_ptr(), X_d.data_ptr(), g_d.data_ptr(),
                               E_d.data_ptr())
    torch.cuda.synchronize()
    Xp[:, :n], gp[:, :n] = X ^ M, want_g
    assert np.array_equal(X_d.cpu().numpy(), Xp) and np.array_equal(g_d.cpu().numpy(), gp)
    assert np.array_equal(E_d.cpu().numpy(), want_E)
