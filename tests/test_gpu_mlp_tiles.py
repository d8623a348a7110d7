"""The network's tiled kernels at the edges of their tiles (16 to 128 rows per
CTA for the scores, chosen by the number of rows; 64 for the gradient)."""
import numpy as np
import pytest

from oracle import mlp_ref as M
from paper_2502_13947_gb300 import icd2s as I
from tests.gpu_util import dev, torch_cuda
from tests.test_gpu_learned import _features, _net, _weights

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 15, 17, 16 * 608 + 1, 32 * 608 + 33, 64 * 608 + 1])
def test_scores_equal_oracle(orc, rows):
    torch_cuda()
    F = _features(rows, rows)
    m, Wb = _net(_weights(2))
    out = dev(np.full(rows + 1, 7.0, np.float32))
    I.icd2s_mlp_score(m, dev(F).data_ptr(), rows, out.data_ptr())
    s = out.cpu().numpy()
    I.icd2s_mlp_destroy(m)
    assert np.array_equal(s[:rows].view(np.uint32), orc.mlp_score_f32(Wb, F).view(np.uint32))
    assert s[rows] == 7.0


def _rounded_products(Wb, F, y, pos_weight):
    """Loss and gradient in 64 bits with h1 and dL/da2 rounded to BF16 as operands of the 64-wide
    products, as the tensor-core gradient is defined.  (At few rows the unrounded reference cannot
    stand in for it: one hidden unit on the other side of its ReLU moves a mean over 64 rows by more
    than the bound.)"""
    W = np.asarray(Wb, np.float64)
    W1, b1, W2 = W[:384].reshape(64, 6), W[384:448], W[448:4544].reshape(64, 64)
    b2, w3, b3 = W[4544:4608], W[4608:4672], W[4672]
    F = np.asarray(F, np.float64)
    rnd = lambda a: M.bf16_round(a.astype(np.float32)).astype(np.float64)
    h1 = rnd(np.maximum(F @ W1.T + b1, 0))
    h2 = np.maximum(h1 @ W2.T + b2, 0)
    s = h2 @ w3 + b3
    sg, n = 1 / (1 + np.exp(-s)), len(F)
    loss = np.mean(pos_weight * y * np.logaddexp(0, -s) + (1 - y) * np.logaddexp(0, s))
    ds = (pos_weight * y * (sg - 1) + (1 - y) * sg) / n
    d2 = ds[:, None] * w3 * (h2 > 0)
    d1 = (rnd(d2) @ W2) * (h1 > 0)
    return loss, np.concatenate([(d1.T @ F).ravel(), d1.sum(0), (rnd(d2).T @ h1).ravel(), d2.sum(0), ds @ h2, [ds.sum()]])


@pytest.mark.parametrize("tc", [False, True])
@pytest.mark.parametrize("rows", [1, 63, 64, 65, 1025])
def test_gradient_matches_reference(rows, tc):
    """The bounds of the library's other gradient tests, for either product."""
    torch = torch_cuda()
    F = _features(rows + 3, rows)
    y = (np.random.default_rng(rows).uniform(size=rows) < 0.5).astype(np.uint8)
    m, Wb = _net(_weights(6))
    I.icd2s_mlp_set_tensor_cores(m, tc)
    grad = torch.zeros(M.NPAR, dtype=torch.float32, device="cuda")
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    Fd, yd = dev(F), dev(y)
    I.icd2s_mlp_grad(m, Fd.data_ptr(), yd.data_ptr(), rows, 3.0, grad.data_ptr(), loss.data_ptr())
    g = grad.cpu().numpy()
    I.icd2s_mlp_destroy(m)
    L_ref, g_ref = (_rounded_products if tc else M.loss_and_grad)(Wb, F, y, 3.0)
    assert abs(float(loss.cpu()[0]) - L_ref) <= (2e-3 if tc else 1e-5) * (1 + abs(L_ref))
    err = np.abs(g - g_ref)
    assert np.all((err <= 1e-3) | (err <= 1e-2 * np.abs(g_ref)))
    if not tc:
        assert np.max(err) <= 1e-4
