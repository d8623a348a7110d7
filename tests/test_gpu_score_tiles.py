"""Scores on both sides of the lines between the tile sizes: 16, 32, 64 and 128 rows per CTA
from 8, 32 and 320 rows per SM on (152 SMs)."""
import numpy as np
import pytest

from paper_2502_13947_gb300 import icd2s as I
from tests.gpu_util import dev, torch_cuda
from tests.test_gpu_learned import _features, _net, _weights

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [63, 8 * 152, 8 * 152 + 1, 32 * 152, 32 * 152 + 1, 320 * 152, 320 * 152 + 1])
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
