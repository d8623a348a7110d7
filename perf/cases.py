"""The workloads that this library's performance is measured on.

Each case is one call, or one short sequence of calls, that a program makes
through the public entry points (include/icd2s.h and its binding): the
evaluation of solutions, whole runs, whole outer iterations of Algorithm 2,
rounds of the Ising machine, the exact Ising machine, the write-back on
caller-owned buffers, and the proposal network's forward and backward.  Sizes
are those of the repository's own workloads (instances.py, bench.py, tests).
"""
from __future__ import annotations

import math

import torch

from paper_2502_13947_gb300 import icd2s as I

_DEV = "cuda"


# --------------------------------------------------------------------------- the cases
def listed():
    return [
        # a handful of candidate solutions of the smallest instance: launches and latency
        dict(name="energy-n64-x8", kind="energy", n=64, density=1.0, count=8),
        # a whole solution set of the dense n = 7000 instance evaluated from scratch
        dict(name="energy-n7000-x256", kind="energy", n=7000, density=1.0, count=256),
        # the whole method on the small dense instance, as a user's first program calls it
        dict(name="run-n64-z8", kind="run", n=64, density=1.0, z=8, m=16, sweeps=256, iters=40, alpha=320, im_mode=0),
        # the flagship: one outer iteration of the sparse n = 2500 instance, host buffers in and out
        dict(name="step-n2500-z128", kind="step", n=2500, density=0.1, z=128, K=1, m_min=64, m_max=64, sweeps=1024,
             alpha=12500, T_max=1500.0, mut_rate=0.01, select_mode=0, use_graph=0, ablation=0, aspiration=0,
             im_order=0),
        # the method that reaches the n = 5000 target first: learned selection, four uneven subQUBOs per
        # solution, the iteration replayed as a CUDA graph
        dict(name="step-n5000-z32-learned", kind="step", n=5000, density=0.5, z=32, K=4, m_min=32, m_max=256,
             sweeps=256, alpha=5000, T_max=2000.0, mut_rate=-1.0, select_mode=1, use_graph=1, ablation=0,
             aspiration=0, im_order=0),
        # one outer iteration of the largest instance of the time-to-target runs
        dict(name="step-n10000-z32", kind="step", n=10000, density=0.5, z=32, K=1, m_min=64, m_max=64, sweeps=256,
             alpha=10000, T_max=2000.0, mut_rate=-1.0, select_mode=0, use_graph=0, ablation=0, aspiration=0,
             im_order=0),
        # the uneven 32-256 batch: Ising-machine rounds on the dense n = 7000 instance and the drift check
        dict(name="rounds-n7000-z256", kind="rounds", n=7000, density=1.0, z=256, K=16, m_min=32, m_max=256,
             sweeps=256, rounds=4),
        # the exact Ising machine at the largest size that it takes, one subQUBO per replica
        dict(name="exact-m24-x128", kind="exact", n=2500, density=0.1, z=128, K=1, m_min=24, m_max=24),
        # the write-back of 1024 flips per solution on the caller's own buffers, at an odd n
        dict(name="writeback-n15999-z16", kind="writeback", n=15999, z=16, flips=1024),
        # scores of every variable of 32 solutions of the n = 10 000 instance
        dict(name="score-320000", kind="score", rows=320000),
        # a gradient of the network over one batch, as a trainer of several workers takes it
        dict(name="grad-8192", kind="grad", rows=8192, tensor_cores=0),
        # training steps of the network on batches of an improvement log
        dict(name="train-8192", kind="train", rows=255256, batch=8192, steps=10, tensor_cores=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["energy", "run", "step", "step", "step", "step", "rounds", "exact", "writeback", "score",
                       "grad", "train"])
    if kind == "energy":
        return dict(kind=kind, n=_log(rng, 33, 7000), density=rng.choice([0.1, 0.5, 1.0]), count=_log(rng, 1, 256))
    if kind == "run":
        n = _log(rng, 40, 400)
        return dict(kind=kind, n=n, density=rng.choice([0.3, 1.0]), z=rng.randint(2, 16), m=rng.randint(8, 20),
                    sweeps=_log(rng, 32, 256), iters=rng.randint(5, 40), alpha=n * rng.choice([1, 5]),
                    im_mode=rng.choice([0, 0, 1]))
    if kind == "step":
        n = _log(rng, 200, 10000)
        K = rng.choice([1, 1, 2, 4, 16]) if n >= 2000 else 1
        m_max = rng.randint(16, 100 if n < 2000 else 256 if K * 256 <= n // 2 else 128)
        m_max = min(m_max, n // (2 * K))
        option = rng.choice(["plain", "plain", "plain", "learned", "hybrid", "no_im", "no_sm", "aspiration",
                             "gauss_seidel"])
        return dict(kind=kind, n=n, density=rng.choice([0.1, 0.5, 1.0]),
                    z=_log(rng, 4, 128 if n <= 3000 else 32), K=K, m_min=rng.randint(8, m_max), m_max=m_max,
                    sweeps=_log(rng, 64, 1024 if K == 1 and n <= 3000 else 256),
                    alpha=n * (rng.choice([1, 5]) if n <= 4000 else 1), T_max=rng.choice([100.0, 1500.0, 2000.0]),
                    mut_rate=rng.choice([-1.0, 0.01, 0.2]),
                    select_mode={"learned": 1, "hybrid": 2}.get(option, 0), use_graph=rng.randint(0, 1),
                    ablation={"no_im": 1, "no_sm": 2}.get(option, 0), aspiration=int(option == "aspiration"),
                    im_order=int(option == "gauss_seidel" and K <= 4))
    if kind == "rounds":
        n = _log(rng, 2000, 7000)
        return dict(kind=kind, n=n, density=rng.choice([0.1, 0.5, 1.0]), z=_log(rng, 16, 256),
                    K=rng.choice([2, 4, n // 512]), m_min=rng.randint(8, 64), m_max=rng.randint(64, 256),
                    sweeps=_log(rng, 64, 256), rounds=rng.randint(2, 6))
    if kind == "exact":
        m = rng.randint(10, 24)
        return dict(kind=kind, n=_log(rng, 200, 5000), density=rng.choice([0.1, 1.0]), z=_log(rng, 4, 128), K=1,
                    m_min=rng.randint(max(1, m - 4), m), m_max=m)
    if kind == "writeback":
        n = _log(rng, 300, 16000)
        return dict(kind=kind, n=n, z=_log(rng, 2, 32), flips=_log(rng, 1, max(2, n // 8)))
    if kind == "score":
        return dict(kind=kind, rows=_log(rng, 1, 320000))
    if kind == "grad":
        return dict(kind=kind, rows=_log(rng, 100, 32768), tensor_cores=rng.randint(0, 1))
    rows = _log(rng, 2000, 255256)
    return dict(kind=kind, rows=rows, batch=_log(rng, 256, 8192), steps=rng.randint(2, 10),
                tensor_cores=rng.randint(0, 1))


# --------------------------------------------------------------------------- inputs
class _Handle:
    """A library handle that is given back when the program drops it."""

    def __init__(self, h, destroy, *keeps):
        self.h, self._destroy, self._keeps = h, destroy, keeps  # _keeps: what this handle refers to

    def __del__(self):
        if self.h is not None:
            self._destroy(self.h)
            self.h = None


def _gen(seed):
    return torch.Generator(device=_DEV).manual_seed(int(seed))


def _matrix(n, density, seed):
    """A symmetric int8 matrix as instances.make_qubo describes it, made on the GPU."""
    g = _gen(seed)
    V = torch.randint(-100, 101, (n, n), generator=g, device=_DEV, dtype=torch.int8)
    if density < 1.0:
        V = torch.where(V == 0, torch.ones_like(V), V)
        V *= torch.rand((n, n), generator=g, device=_DEV, dtype=torch.float32) < density
    U = torch.triu(V)
    return U + torch.triu(U, 1).T


def _qubo(n, density, seed):
    Q = _matrix(n, density, seed).cpu().numpy()
    return _Handle(I.icd2s_qubo_create(Q), I.icd2s_qubo_destroy)


def _solutions(n, count, seed):
    return torch.randint(0, 2, (count, n), generator=_gen(seed + 1), device=_DEV, dtype=torch.uint8)


def _tenure(n):
    return max(2, n // 150)


def _features(rows, seed):
    """Feature rows of the kind that the search produces, and labels of which about one in twelve is set."""
    g = _gen(seed + 2)
    r = torch.rand((rows, 6), generator=g, device=_DEV, dtype=torch.float32)
    F = torch.empty((rows, 6), device=_DEV, dtype=torch.float32)
    F[:, 0] = (r[:, 0] < 0.5).float()             # x
    F[:, 1] = r[:, 1] * 2 - 0.4                   # g / (max |g| + 1)
    F[:, 2] = r[:, 2] ** 6 * 0.02                 # toggles / alpha
    F[:, 3] = (r[:, 3] - 0.9).clamp(min=0) * 10   # tabu memory / c
    F[:, 4] = r[:, 4] ** 3                        # hits / (t + 1)
    F[:, 5] = 0.85 + 0.15 * r[:, 5]               # eta_hat
    y = (torch.rand(rows, generator=g, device=_DEV) < 0.02 + 0.25 * F[:, 2] * 50 * F[:, 0]).to(torch.uint8)
    return F, y


def _pinned(shape, dtype):
    return torch.empty(shape, dtype=dtype, pin_memory=True).numpy()


def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case)
    if kind == "energy":
        s["q"] = _qubo(case["n"], case["density"], seed)
        s["x"] = _solutions(case["n"], case["count"], seed)
        s["E"] = torch.empty(case["count"], device=_DEV, dtype=torch.int64)
    elif kind == "run":
        n = case["n"]
        s["q"] = _qubo(n, case["density"], seed)
        s["seed"] = int(seed)
        s["p"] = I.icd2s_default_params(n, z=case["z"], m_min=case["m"], m_max=case["m"], m_init=case["m"],
                                        alpha=case["alpha"], c=_tenure(n), sweeps=case["sweeps"], patience=0,
                                        max_iters=case["iters"], im_mode=case["im_mode"])
    elif kind == "step":
        n, z = case["n"], case["z"]
        q = _qubo(n, case["density"], seed)
        st = s["st"] = _Handle(I.icd2s_state_create(q.h, z, int(seed)), I.icd2s_state_destroy, q)
        const = case["mut_rate"] >= 0
        s["p"] = I.icd2s_default_params(
            n, z=z, K=case["K"], m_min=case["m_min"], m_max=case["m_max"], m_init=min(case["m_max"], n),
            alpha=case["alpha"], c=_tenure(n), sweeps=case["sweeps"], T_max=case["T_max"], T_min=1.0, patience=0,
            mut_mode=1 if const else 0, mut_rate=case["mut_rate"] if const else 0.0, use_graph=case["use_graph"],
            select_mode=case["select_mode"], ablation=case["ablation"], aspiration=case["aspiration"],
            im_order=case["im_order"])
        if case["select_mode"]:
            s["mlp"] = _Handle(I.icd2s_mlp_create(int(seed)), I.icd2s_mlp_destroy)
            I.icd2s_state_set_mlp(st.h, s["mlp"].h)
        s["x_in"], s["x_out"] = _pinned((z, n), torch.uint8), _pinned((z, n), torch.uint8)
        s["E"] = _pinned((z,), torch.int64)
        # the solutions that iteration 1 starts from: those that iteration 0 left
        s["x_in"][:] = _solutions(n, z, seed).cpu().numpy()
        I.icd2s_step_host(st.h, s["p"], 0, s["x_in"], s["x_out"], s["E"], _stream())
        s["x_in"][:] = s["x_out"]
    elif kind == "rounds":
        n, z = case["n"], case["z"]
        q = _qubo(n, case["density"], seed)
        st = s["st"] = _Handle(I.icd2s_state_create(q.h, z, int(seed)), I.icd2s_state_destroy, q)
        s["p"] = I.icd2s_default_params(n, z=z, K=case["K"], m_min=case["m_min"], m_max=case["m_max"],
                                        c=_tenure(n), sweeps=case["sweeps"], T_max=2000.0, T_min=1.0)
        I.icd2s_tabu(st.h, n // 2, _tenure(n), _stream())   # a round follows a Tabu search
        s["x_out"], s["E"] = _pinned((z, n), torch.uint8), _pinned((z,), torch.int64)
        I.icd2s_get_state(st.h, z, n, s["x_out"], s["E"], want_g=False)
        s["x_in"] = torch.from_numpy(s["x_out"]).to(_DEV)
    elif kind == "exact":
        n, z, K = case["n"], case["z"], case["K"]
        q = _qubo(n, case["density"], seed)
        st = s["st"] = _Handle(I.icd2s_state_create(q.h, z, int(seed)), I.icd2s_state_destroy, q)
        I.icd2s_tabu(st.h, n // 2, _tenure(n), _stream())
        s["idx"] = torch.zeros(z * K * case["m_max"] + 1, device=_DEV, dtype=torch.int32)
        s["off"] = torch.zeros(z * K + 1, device=_DEV, dtype=torch.int32)
        sp = I.SelectParams(w1=65536, w2=65536, w3=32768, K=K, m_min=case["m_min"], m_max=case["m_max"], iter=0)
        I.icd2s_select_subqubos(st.h, sp, s["idx"].data_ptr(), s["off"].data_ptr(), _stream())
        s["flips"] = torch.zeros((z, n), device=_DEV, dtype=torch.uint8)
        s["dE"] = torch.zeros(z * K, device=_DEV, dtype=torch.int64)
    elif kind == "writeback":
        n, z = case["n"], case["z"]
        ld = (n + 127) // 128 * 128
        s["ld"] = ld
        Q = torch.zeros((n, ld), device=_DEV, dtype=torch.int8)
        Q[:, :n] = _matrix(n, 1.0, seed)
        x = torch.zeros((z, ld), device=_DEV, dtype=torch.uint8)
        x[:, :n] = _solutions(n, z, seed)
        g, E = _gains(Q, x, n)
        s["flips"] = _flips(n, z, case["flips"], seed)
        s["Q"], s["x"], s["g"], s["E"] = Q, x, g.to(torch.int32), E
    else:
        rows = case["rows"]
        s["F"], s["y"] = _features(rows, seed)
        s["mlp"] = _Handle(I.icd2s_mlp_create(int(seed)), I.icd2s_mlp_destroy)
        if kind == "score":
            s["out"] = torch.empty(rows, device=_DEV, dtype=torch.float32)
        else:
            I.icd2s_mlp_set_tensor_cores(s["mlp"].h, bool(case["tensor_cores"]))
            s["W"] = I.icd2s_mlp_get_weights(s["mlp"].h)[0]
            s["grad"] = torch.empty(I.MLP_PARAMS, device=_DEV, dtype=torch.float32)
            s["loss"] = torch.empty(1, device=_DEV, dtype=torch.float32)
    return s


def _gains(Q, x, n):
    """Gains [z][ld] (padding 0) and energies [z] of the rows of x, exact: every sum is below 2^24."""
    z, ld = x.shape
    xf = x[:, :n].float()
    h = torch.empty((z, n), device=_DEV, dtype=torch.float32)
    for a in range(0, n, 4096):
        h[:, a:a + 4096] = xf @ Q[a:a + 4096, :n].float().T
    d = torch.diagonal(Q[:, :n]).float()
    off = h - xf * d
    g = torch.zeros((z, ld), device=_DEV, dtype=torch.float64)
    g[:, :n] = ((1 - 2 * xf) * (d + 2 * off)).double()
    E = (xf.double() * (d + off).double()).sum(1).to(torch.int64)
    return g, E


def _flips(n, z, flips, seed):
    """0/1 masks [z][n] with `flips` set positions in each row."""
    order = torch.argsort(torch.rand((z, n), generator=_gen(seed + 3), device=_DEV), dim=1)
    m = torch.zeros((z, n), device=_DEV, dtype=torch.uint8)
    m.scatter_(1, order[:, :flips], 1)
    return m


# --------------------------------------------------------------------------- one pass
def run(s):
    kind, sp = s["kind"], _stream()
    if kind == "energy":
        I.icd2s_energy(s["q"].h, s["x"].data_ptr(), s["count"], s["E"].data_ptr(), sp)
        return {"E": s["E"]}
    if kind == "run":
        r = I.icd2s_run(s["q"].h, s["p"], s["seed"], want_S=True)
        return {"x": r["best_x"], "E": r["best_E"], "S": r["S"]}
    if kind == "step":
        if s["select_mode"]:  # icd2s_state_load also clears the hit counts that the network reads
            I.icd2s_state_load(s["st"].h, s["x_in"], stream=sp)
            I.icd2s_step_host(s["st"].h, s["p"], 1, None, s["x_out"], s["E"], sp)
        else:
            I.icd2s_step_host(s["st"].h, s["p"], 1, s["x_in"], s["x_out"], s["E"], sp)
        return {"x": s["x_out"], "E": s["E"]}
    if kind == "rounds":
        st = s["st"].h
        I.icd2s_state_load(st, s["x_in"].data_ptr(), x_is_device=True, stream=sp)
        for t in range(s["rounds"]):
            I.icd2s_im_round(st, s["p"], t, sp)
        bad = I.icd2s_refresh(st, stream=sp)
        I.icd2s_get_state(st, s["z"], s["n"], s["x_out"], s["E"], want_g=False)
        return {"x": s["x_out"], "E": s["E"], "mismatches": bad}
    if kind == "exact":
        I.icd2s_exact_subqubos_batch(s["st"].h, s["idx"].data_ptr(), s["off"].data_ptr(), s["z"] * s["K"], s["K"],
                                     s["flips"].data_ptr(), s["dE"].data_ptr(), sp)
        return {"flips": s["flips"], "dE": s["dE"]}
    if kind == "writeback":
        I.icd2s_apply_flips_static(s["Q"].data_ptr(), s["n"], s["ld"], s["z"], s["flips"].data_ptr(),
                                   s["x"].data_ptr(), s["g"].data_ptr(), s["E"].data_ptr(), sp)
        return {"x": s["x"], "g": s["g"], "E": s["E"]}
    m = s["mlp"].h
    if kind == "score":
        I.icd2s_mlp_score(m, s["F"].data_ptr(), s["rows"], s["out"].data_ptr(), sp)
        return {"score": s["out"]}
    if kind == "grad":
        I.icd2s_mlp_grad(m, s["F"].data_ptr(), s["y"].data_ptr(), s["rows"], 10.0, s["grad"].data_ptr(),
                         s["loss"].data_ptr(), sp)
        return {"grad": s["grad"], "loss": s["loss"]}
    I.icd2s_mlp_set_weights(m, s["W"])
    loss = I.icd2s_mlp_train(m, s["F"].data_ptr(), s["y"].data_ptr(), s["rows"], s["steps"], s["batch"], lr=2e-3,
                             pos_weight=10.0, stream=sp)
    return {"weights": I.icd2s_mlp_get_weights(m)[0], "loss": loss}


# --------------------------------------------------------------------------- what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind == "energy":
        n, r = case["n"], case["count"]
        return {"bytes": n * n + r * n + 8 * r, "flops": 2 * n * n * r}
    if kind in ("run", "step"):
        n, z = case["n"], case["z"]
        if kind == "run":
            its, attempts = case["iters"], case["z"] * case["m"] * case["sweeps"]
            attempts = 0 if case["im_mode"] else attempts + attempts * (n // case["m"]) // case["iters"]
        else:
            its = 1
            attempts = 0 if case["ablation"] == 1 else (
                z * case["K"] * (case["m_min"] + case["m_max"]) // 2 * case["sweeps"])
        # per Tabu move one multiply-add and one comparison per variable; per attempt one comparison
        return {"bytes": n * n + 2 * z * n + 8 * z, "flops": its * (z * case["alpha"] * 3 * n + attempts)}
    if kind == "rounds":
        n, z = case["n"], case["z"]
        attempts = z * case["K"] * (case["m_min"] + case["m_max"]) // 2 * case["sweeps"] * case["rounds"]
        return {"bytes": n * n + 2 * z * n + 8 * z, "flops": attempts + 2 * n * n * z}
    if kind == "exact":
        s = case["z"] * case["K"]
        m = (case["m_min"] + case["m_max"]) / 2
        return {"bytes": s * (m * m + 5 * m + 8) + case["z"] * case["n"], "flops": s * 2 * 2 ** case["m_max"]}
    if kind == "writeback":
        n, z, f = case["n"], case["z"], case["flips"]
        rows = n * (1 - (1 - f / n) ** z)   # the rows of Q that some solution flips, each read once
        return {"bytes": rows * n + z * (n + 10 * n + 16), "flops": 2 * z * f * n}
    if kind == "score":
        return {"bytes": case["rows"] * 28 + 2 * I.MLP_PARAMS, "flops": case["rows"] * 2 * (384 + 4096 + 64)}
    rows, steps = (case["rows"], 1) if kind == "grad" else (min(case["batch"], case["rows"]), case["steps"])
    return {"bytes": steps * (rows * 25 + 14 * I.MLP_PARAMS), "flops": steps * rows * 6 * (384 + 4096 + 64)}


# --------------------------------------------------------------------------- the same in 64 bits
def _bf16_weights(seed):
    """The network's weights as it computes with them (its own random start, rounded to BF16), in 64 bits."""
    m = _Handle(I.icd2s_mlp_create(int(seed)), I.icd2s_mlp_destroy)
    W = torch.from_numpy(I.icd2s_mlp_get_weights(m.h)[0]).bfloat16().double().to(_DEV)
    return W[:384].view(64, 6), W[384:448], W[448:4544].view(64, 64), W[4544:4608], W[4608:4672], W[4672:]


def exact(case, seed):
    kind = case["kind"]
    if kind == "energy":
        n = case["n"]
        Q, x = _matrix(n, case["density"], seed).double(), _solutions(n, case["count"], seed).double()
        return {"E": ((x @ Q) * x).sum(1)}
    if kind == "writeback":
        n, z = case["n"], case["z"]
        Q = _matrix(n, 1.0, seed)
        x = torch.zeros((z, (n + 127) // 128 * 128), device=_DEV, dtype=torch.uint8)
        x[:, :n] = _solutions(n, z, seed) ^ _flips(n, z, case["flips"], seed)
        g, E = _gains(Q, x, n)
        return {"x": x.double(), "g": g, "E": E.double()}
    if kind in ("score", "grad"):
        F, y = _features(case["rows"], seed)
        P = [w.clone().requires_grad_(kind == "grad") for w in _bf16_weights(seed)]
        F, y = F.double(), y.double()
        h = torch.relu(F @ P[0].T + P[1])
        h = torch.relu(h @ P[2].T + P[3])
        s = h @ P[4] + P[5]
        if kind == "score":
            return {"score": s}
        sp = torch.nn.functional.softplus
        loss = (10.0 * y * sp(-s) + (1 - y) * sp(s)).mean()
        loss.backward()
        return {"grad": torch.cat([w.grad.reshape(-1) for w in P]), "loss": loss.detach().reshape(1)}
    # the solver's other outputs are whole numbers; a trained network's weights are rounded to BF16 at
    # every step, where a difference in the last bit may move a weight by 0.4 %
    return None
