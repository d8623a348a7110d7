"""Energies and recomputed gains when the tensor-core product's pipeline times out: the
plain product replaces sums that some tiles have added and others have not."""
import numpy as np
import pytest

from paper_2502_13947_gb300 import icd2s as I
from paper_2502_13947_gb300.instances import make_qubo, random_solutions
from tests.gpu_util import dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,rows", [(513, 1), (700, 129), (1153, 33), (1500, 257), (2501, 3)])
def test_timed_out_product_gives_the_exact_values(n, rows):
    torch = torch_cuda()
    Q = make_qubo(n, 1.0, n, lo=-128, hi=127)
    X = random_solutions(n, rows, 3)
    X[0] = 1
    Qf, Xf = Q.astype(np.float64), X.astype(np.float64)
    H, d = Xf @ Qf, np.diag(Qf)
    E = (H * Xf).sum(1).astype(np.int64)
    G = ((1 - 2 * Xf) * (d + 2 * (H - Xf * d))).astype(np.int64)
    x_d, E_d = dev(X), torch.empty(rows, dtype=torch.int64, device="cuda")
    q = I.icd2s_qubo_create(Q)
    times = []
    for stalls in (0, 1, 0):   # the last call runs normally again
        E_d.fill_(7)
        I.icd2s_debug_product_stall(q, stalls, 20000)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        I.icd2s_energy(q, x_d.data_ptr(), rows, E_d.data_ptr(), torch.cuda.current_stream().cuda_stream)
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b))
        assert np.array_equal(E_d.cpu().numpy(), E)
    assert times[1] > 20.0 > times[2]   # ms: the stalled tiles waited their 20 ms
    I.icd2s_debug_product_stall(q, 2, 2000)
    st = I.icd2s_state_create(q, rows, 5)   # the first product, of the initial set
    x0, g0, e0 = I.icd2s_get_state(st, rows, n)
    xf = x0.astype(np.float64)
    h = xf @ Qf
    assert np.array_equal(e0, (h * xf).sum(1).astype(np.int64))
    assert np.array_equal(g0, ((1 - 2 * xf) * (d + 2 * (h - xf * d))).astype(np.int64))
    for _ in range(2):                      # the second product stalls, the third does not
        I.icd2s_state_load(st, X)
        x, g, e = I.icd2s_get_state(st, rows, n)
        assert np.array_equal(x, X) and np.array_equal(g, G) and np.array_equal(e, E)
    I.icd2s_state_destroy(st)
    I.icd2s_qubo_destroy(q)
