"""The annealer's decisions by blocks of 32 positions where they hang on one another:
chains in which every accept makes the next one possible (a block then takes as many
rounds as it has positions), cold dense subQUBOs, and uneven batches on both sides of the
size classes' limits."""
import numpy as np
import pytest

from paper_2502_13947_gb300 import icd2s as I
from paper_2502_13947_gb300.instances import make_qubo, random_solutions, random_subsets
from tests.gpu_util import dev, lib_params, torch_cuda
from tests.test_gpu_run import _compare_runs

pytestmark = pytest.mark.gpu

SIZES = [31, 32, 33, 63, 64, 65, 127, 128, 129, 191, 192, 193, 255, 256]


def _chain(n):
    """x = 0: position 0 goes downhill, every other one only once its predecessor is 1."""
    Q = np.zeros((n, n), np.int8)
    i = np.arange(n - 1)
    Q[i, i + 1] = Q[i + 1, i] = -100
    np.fill_diagonal(Q, 100)
    Q[0, 0] = -1
    return Q


@pytest.mark.parametrize("m", SIZES)
@pytest.mark.parametrize("kind", ["chain", "cold"])
def test_dependent_decisions(orc, m, kind):
    torch = torch_cuda()
    n, it, sweeps = 600, 5, 6
    Q = _chain(n) if kind == "chain" else make_qubo(n, 1.0, 8, lo=-128, hi=127)
    X = np.zeros((1, n), np.uint8) if kind == "chain" else random_solutions(n, 1, 2)
    S = np.arange(m, dtype=np.int32) if kind == "chain" else np.sort(random_subsets(n, [m], m)).astype(np.int32)
    T = 0.01 if kind == "chain" else 40.0
    q = I.icd2s_qubo_create(Q)
    st = I.icd2s_state_create(q, 1, 77)
    I.icd2s_state_load(st, X)
    mask, dE = torch.zeros((1, n), dtype=torch.uint8, device="cuda"), torch.zeros(1, dtype=torch.int64, device="cuda")
    idx_d, off_d = dev(S), dev(np.array([0, m], np.int32))
    ap = I.AnnealParams(sweeps=sweeps, T_max=T, T_min=T, iter=it, per_replica=1)
    I.icd2s_anneal_subqubos_batch(st, idx_d.data_ptr(), off_d.data_ptr(), 1, ap, mask.data_ptr(), dE.data_ptr())
    Qs, _ = orc.subqubo(Q, X[0], S)
    want, dE_o, _ = orc.anneal(Qs, X[0][S], orc.beta_table(sweeps, T, T), orc.nlog_table(), 77, 0, it)
    got = X[0] ^ mask.cpu().numpy()[0]
    if kind == "chain":
        assert want.all()   # the whole chain follows within the first sweep
    assert np.array_equal(got[S], want) and int(dE.cpu()[0]) == dE_o
    I.icd2s_state_destroy(st)
    I.icd2s_qubo_destroy(q)


@pytest.mark.parametrize("m_min,m_max", [(24, 40), (56, 72), (120, 136), (184, 200), (40, 256)])
def test_cold_uneven_batches(orc, m_min, m_max):
    n = 1100
    Q = make_qubo(n, 1.0, 9, lo=-128, hi=127)
    lp = lib_params(I, n, z=3, K=4, m_min=m_min, m_max=m_max, m_init=m_max, alpha=200, c=4, sweeps=12, T_max=60.0,
                    T_min=0.5, mut_mode=1, mut_rate=0.3, patience=0, max_iters=3)
    _compare_runs(orc, Q, lp, 13)
