"""The write-back at the edges of its split: list lengths around the four rows
added at a time and the 2048 staged ones, one to eight CTAs per tile (many or
few solutions), 16- and 4-byte row loads."""
import numpy as np
import pytest

from paper_2502_13947_gb300 import icd2s as I
from paper_2502_13947_gb300.instances import make_qubo, random_solutions
from tests.gpu_util import dev, torch_cuda

pytestmark = pytest.mark.gpu


def _state(Q, X):
    Qf, Xf = Q.astype(np.float64), X.astype(np.float64)
    H, d = Xf @ Qf, np.diag(Qf)
    return (((1 - 2 * Xf) * (d + 2 * (H - Xf * d))).astype(np.int64), (H * Xf).sum(1).astype(np.int64))


@pytest.mark.parametrize("n,R,ld", [(2500, 3, 2500), (2500, 3, 2560), (300, 200, 384), (300, 700, 300), (4100, 1, 4224)])
def test_lists_of_every_length(n, R, ld):
    torch = torch_cuda()
    Q = make_qubo(n, 1.0, 3, lo=-128, hi=127)
    X = random_solutions(n, R, 4)
    lengths = [0, 1, 3, 4, 5, 15, 16, 17, 63, 64, 65, 255, 257, 300, n // 2, n - 1, n]
    rng = np.random.default_rng(1)
    M = np.zeros((R, n), np.uint8)
    for p in range(R):
        M[p, rng.permutation(n)[:min(n, lengths[(5 * p + (16 if R < 4 else 0)) % len(lengths)])]] = 1
    g, E = _state(Q, X)
    want_g, want_E = _state(Q, X ^ M)
    # the handle's path
    q = I.icd2s_qubo_create(Q)
    st = I.icd2s_state_create(q, R, 1)
    I.icd2s_state_load(st, X)
    M_d = dev(M)
    I.icd2s_apply_flips_update_gains(st, M_d.data_ptr())
    x1, g1, e1 = I.icd2s_get_state(st, R, n)
    assert np.array_equal(x1, X ^ M) and np.array_equal(g1, want_g) and np.array_equal(e1, want_E)
    I.icd2s_state_destroy(st)
    I.icd2s_qubo_destroy(q)
    # the caller's buffers
    Qp, Xp, gp = np.zeros((n, ld), np.int8), np.full((R, ld), 7, np.uint8), np.full((R, ld), -5, np.int32)
    Qp[:, :n], Xp[:, :n], gp[:, :n] = Q, X, g
    Q_d, X_d, g_d, E_d = dev(Qp), dev(Xp), dev(gp), dev(E)
    I.icd2s_apply_flips_static(Q_d.data_ptr(), n, ld, R, M_d.data_ptr(), X_d.data_ptr(), g_d.data_ptr(),
                               E_d.data_ptr())
    torch.cuda.synchronize()
    Xp[:, :n], gp[:, :n] = X ^ M, want_g
    assert np.array_equal(X_d.cpu().numpy(), Xp) and np.array_equal(g_d.cpu().numpy(), gp)
    assert np.array_equal(E_d.cpu().numpy(), want_E)
