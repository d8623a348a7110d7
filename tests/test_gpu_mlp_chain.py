"""Training steps launched ahead of one another against the same steps one call at a
time (the first step of a call is never launched ahead)."""
import numpy as np
import pytest

from paper_2502_13947_gb300 import icd2s as I
from tests.gpu_util import dev, torch_cuda
from tests.test_gpu_learned import _features

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tc", [False, True])
@pytest.mark.parametrize("rows,batch,steps", [(700, 64, 300), (20000, 8192, 200), (3000, 3000, 100)])
def test_chained_steps_equal_single_ones(rows, batch, steps, tc):
    """Weights and losses bit for bit: both sides add in the same fixed order."""
    torch_cuda()
    F_d = dev(_features(rows, rows))
    y_d = dev((np.random.default_rng(rows).uniform(size=rows) < 0.3).astype(np.uint8))
    got = []
    for parts in ([steps], [1] * steps):
        m = I.icd2s_mlp_create(5)
        I.icd2s_mlp_set_tensor_cores(m, tc)
        loss = [I.icd2s_mlp_train(m, F_d.data_ptr(), y_d.data_ptr(), rows, k, batch, lr=1e-2, pos_weight=2.0)
                for k in parts]
        got.append([np.concatenate(loss), *I.icd2s_mlp_get_weights(m)])
        I.icd2s_mlp_destroy(m)
    for a, b in zip(*got):
        assert np.array_equal(a.view(np.uint32), b.view(np.uint32))
