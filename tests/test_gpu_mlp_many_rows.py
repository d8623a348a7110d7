"""The gradient over more rows than one launch takes: its scratch stays bounded and its
value stays the mean over all rows."""
import numpy as np
import pytest

from oracle import mlp_ref as M
from paper_2502_13947_gb300 import icd2s as I
from tests.gpu_util import torch_cuda
from tests.test_gpu_learned import _net, _weights

pytestmark = pytest.mark.gpu


def _rows(torch, rows):
    g = torch.Generator(device="cuda").manual_seed(rows)
    F = torch.rand((rows, 6), generator=g, device="cuda")
    y = (torch.rand(rows, generator=g, device="cuda") < 0.2).to(torch.uint8)
    return F, y


def _grad(torch, m, F, y):
    g, L = torch.zeros(M.NPAR, device="cuda"), torch.zeros(1, device="cuda")
    I.icd2s_mlp_grad(m, F.data_ptr(), y.data_ptr(), len(y), 3.0, g.data_ptr(), L.data_ptr())
    torch.cuda.synchronize()
    return g, L


@pytest.mark.parametrize("tc", [False, True])
@pytest.mark.parametrize("rows", [262144, 262145, 2 * 262144 + 63])
def test_gradient_of_many_rows_matches_reference(rows, tc):
    """The bounds of the library's other gradient tests, against 64 bits on the GPU."""
    torch = torch_cuda()
    F, y = _rows(torch, rows)
    m, Wb = _net(_weights(6))
    I.icd2s_mlp_set_tensor_cores(m, tc)
    grad, loss = _grad(torch, m, F, y)
    I.icd2s_mlp_destroy(m)
    W = torch.tensor(np.asarray(Wb, np.float64), device="cuda", requires_grad=True)
    h = torch.relu(F.double() @ W[:384].reshape(64, 6).T + W[384:448])
    h = torch.relu(h @ W[448:4544].reshape(64, 64).T + W[4544:4608])
    s, t = h @ W[4608:4672] + W[4672], y.double()
    ref = (3.0 * t * torch.nn.functional.softplus(-s) + (1 - t) * torch.nn.functional.softplus(s)).mean()
    ref.backward()
    ref = ref.detach()
    assert abs(float(loss[0]) - float(ref)) <= (2e-3 if tc else 1e-5) * (1 + abs(float(ref)))
    err = (grad.double() - W.grad).abs()
    assert bool(((err <= 1e-3) | (err <= 1e-2 * W.grad.abs())).all())
    if not tc:
        assert float(err.max()) <= 1e-4


def test_scratch_does_not_grow_with_the_rows():
    """20 M rows: a partial gradient for every 128 rows would be 2.9 GB."""
    torch = torch_cuda()
    F, y = _rows(torch, 20_000_000)
    m, _ = _net(_weights(6))
    _grad(torch, m, F[:64], y[:64])
    before = torch.cuda.mem_get_info()[0]
    _grad(torch, m, F, y)
    used = before - torch.cuda.mem_get_info()[0]
    I.icd2s_mlp_destroy(m)
    assert used <= 1 << 28, used
