"""The work that users of the solver have it do, as measurable cases: whole
calls of the public entry points on the workloads of ``workloads.py`` and
``bench.py`` (drawn on the GPU here, from the same distributions), from the
smallest batch to the largest.

A case is a dict of plain values.  ``call`` says which entry point it goes
through: "solve" (lp_batch_solve + lp_batch_results), "host" (lp_solve_host),
"noalloc" (lp_solve_uniform_noalloc), "warm" (lp_batch_solve_warm), "train"
(Mlp.train_step) or "hyperbox" (lp_hyperbox_solve); ``family`` which LPs.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1802_08557_gb300 import lpbatch as lpb

F64 = torch.float64


def listed():
    return [
        # the smallest batch: a thousand 5 x 5 LPs, where launches and latency are all there is
        {"name": "fp64_5x5_1k", "call": "solve", "family": "positive", "precision": "fp64", "num": 1000, "m": 5, "n": 5},
        # dense random LPs, a fifth of them with phase I, in plain double precision (the paper's arithmetic)
        {"name": "fp64_50x50_20k", "call": "solve", "family": "mixed_sign", "precision": "fp64", "num": 20_000,
         "m": 50, "n": 50},
        # the benchmark's headline: the same LPs, a full batch, FP32 tableau with the FP64 certificate
        {"name": "mixed_50x50_100k", "call": "solve", "family": "mixed_sign", "precision": "mixed", "num": 100_000,
         "m": 50, "n": 50},
        # reachability: the support function of one polytope of 40 halfspaces in R^10 (x = x+ - x-) in 1e5 directions
        {"name": "mixed_support_40x10_100k", "call": "solve", "family": "support", "precision": "mixed",
         "num": 100_000, "m": 40, "n": 20},
        # LPs of every size from 10 to 500 rows and columns in one batch, full size, double precision
        {"name": "fp64_uneven_20k", "call": "solve", "family": "uneven", "precision": "fp64", "num": 20_000,
         "m": 500, "n": 500, "lo": 10},
        # the same sizes in a smaller batch, mixed precision
        {"name": "mixed_uneven_2k", "call": "solve", "family": "uneven", "precision": "mixed", "num": 2000,
         "m": 500, "n": 500, "lo": 10},
        # one call from pinned host arrays to host results: copies, planning and solve
        {"name": "host_50x50_25k", "call": "host", "family": "mixed_sign", "precision": "mixed", "num": 25_000,
         "m": 50, "n": 50},
        # a loop that must not allocate: equal-size LPs in the caller's own device buffers
        {"name": "noalloc_50x50_1500", "call": "noalloc", "family": "mixed_sign", "precision": "fp64", "num": 1500,
         "m": 50, "n": 50},
        # a parametric family (one shared A) solved from a trained network's proposal
        {"name": "warm_200x100_100k", "call": "warm", "family": "shared", "precision": "fp64", "num": 100_000,
         "m": 200, "n": 100},
        # training that network: steps of 1024 LPs, then the weights back on the host
        {"name": "train_1024", "call": "train", "batch": 1024, "m": 200, "n": 100, "hidden": 512, "steps": 8},
        # box LPs of the paper's 28-variable helicopter model: one box, four million directions, optima only
        {"name": "hyperbox_28_4m", "call": "hyperbox", "num": 1 << 22, "dim": 28, "per_lp": False, "with_x": False},
        # box LPs of its 5-dimensional system: a box per direction, the maximisers wanted too
        {"name": "hyperbox_5_boxes_2m", "call": "hyperbox", "num": 2_000_001, "dim": 5, "per_lp": True, "with_x": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["solve"] * 6 + ["host", "noalloc", "warm", "train", "hyperbox", "hyperbox"])
    if call == "hyperbox":
        dim = _log(rng, 2, 160)
        per_lp, with_x = rng.random() < 0.4, rng.random() < 0.5
        return {"call": call, "num": _log(rng, 1000, (1 << 26) // dim), "dim": dim, "per_lp": per_lp, "with_x": with_x}
    if call == "train":
        return {"call": call, "batch": _log(rng, 100, 1024), "m": _log(rng, 20, 200), "n": _log(rng, 10, 100),
                "hidden": _log(rng, 64, 512), "steps": rng.randint(2, 8)}
    if call == "warm":
        return {"call": call, "family": "shared", "precision": "fp64", "num": _log(rng, 2000, 60_000),
                "m": _log(rng, 60, 200), "n": _log(rng, 30, 100)}
    family = rng.choice(["positive", "mixed_sign", "mixed_sign", "support", "uneven", "uneven"])
    precision = "fp64" if call == "noalloc" else rng.choice(["fp64", "mixed"])
    if call == "noalloc":
        family = rng.choice(["positive", "mixed_sign"])
    if call == "host":
        family = rng.choice(["positive", "mixed_sign", "uneven"])
    if family == "uneven":
        return {"call": call, "family": family, "precision": precision, "num": _log(rng, 100, 4000),
                "m": _log(rng, 60, 500), "n": _log(rng, 60, 500), "lo": rng.randint(5, 20)}
    if family == "support":
        dim = rng.randint(2, 16)
        return {"call": call, "family": family, "precision": precision, "num": _log(rng, 500, 60_000),
                "m": 4 * dim + rng.randint(8, 16), "n": 2 * dim}
    m, n = _log(rng, 4, 130), _log(rng, 4, 130)
    # about m + n pivots of m * n each at most: no more than the largest listed batch
    most = min(100_000, int(8e9 / (m * n * (m + n))), int(1.2e8 / (m * n)), 8000 if call != "solve" else 100_000)
    return {"call": call, "family": family, "precision": precision, "num": _log(rng, 50, max(200, most)), "m": m, "n": n}


# ---------------------------------------------------------------------------
# Inputs, on the GPU
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 2 + 1)


def _uniform(g, lo, hi, *shape):
    return torch.rand(shape, generator=g, device="cuda", dtype=F64) * (hi - lo) + lo


def _sizes(case):
    """Rows and columns of every LP: the case's own, or spread over the logarithm of its range (the same for every seed)."""
    N = case["num"]
    if case["family"] == "uneven":
        lo = case["lo"]
        rs = np.random.RandomState(N + 7 * lo)
        m = np.floor(np.exp(rs.uniform(math.log(lo), math.log(case["m"]), N))).astype(np.int32)
        n = np.floor(np.exp(rs.uniform(math.log(lo), math.log(case["n"]), N))).astype(np.int32)
        return m, n
    return np.full(N, case["m"], np.int32), np.full(N, case["n"], np.int32)


def _offsets(counts):
    o = np.zeros(len(counts), np.int64)
    np.cumsum(counts[:-1].astype(np.int64), out=o[1:])
    return o


def _batch(case, seed):
    """m, n (host), offsets (host) and A, b, c (device, flat) of a case's LPs."""
    g = _gen(seed)
    N, fam = case["num"], case["family"]
    m, n = _sizes(case)
    mn = m.astype(np.int64) * n
    a_off, b_off, c_off = _offsets(mn), _offsets(m), _offsets(n)
    M, K = case["m"], case["n"]
    if fam == "positive":
        A, b, c = _uniform(g, 1.0, 10.0, N, M, K), _uniform(g, 10.0, 100.0, N, M), _uniform(g, 1.0, 10.0, N, K)
    elif fam == "uneven":
        A = torch.rand(int(mn.sum()), generator=g, device="cuda", dtype=F64)
        b = _uniform(g, 1.0, 100.0, int(m.sum()))
        c = _uniform(g, 0.0, 1.0, int(n.sum()))
    elif fam == "support":
        dim = K // 2
        a = torch.randn((M, dim), generator=g, device="cuda", dtype=F64)
        a /= a.norm(dim=1, keepdim=True)
        b = _uniform(g, 1.0, 2.0, M)
        l = torch.randn((N, dim), generator=g, device="cuda", dtype=F64)
        l /= l.norm(dim=1, keepdim=True)
        A, c = torch.cat([a, -a], 1), torch.cat([l, -l], 1)
        a_off, b_off = np.zeros(N, np.int64), np.zeros(N, np.int64)
    elif fam == "shared":
        A, b0 = _uniform(g, 0.0, 1.0, M, K), _uniform(g, 1.0, 100.0, M)
        b = b0 * (1.0 + 0.1 * torch.randn((N, M), generator=g, device="cuda", dtype=F64))
        c = _uniform(g, 0.0, 1.0, N, K)
        a_off = np.zeros(N, np.int64)
    else:
        # random signs: a fifth draws b of both signs (phase I), a fortieth each
        # is infeasible or unbounded by construction
        u = torch.rand(N, generator=g, device="cuda", dtype=F64)
        A, c = _uniform(g, -1.0, 1.0, N, M, K), _uniform(g, -1.0, 1.0, N, K)
        b = torch.where((u < 0.2)[:, None], _uniform(g, -5.0, 10.0, N, M), _uniform(g, 1.0, 10.0, N, M))
        if M >= 2:
            q = torch.nonzero((u >= 0.2) & (u < 0.225)).flatten()
            j = torch.randint(0, M, (N,), generator=g, device="cuda")[q]
            k = (j + 1 + torch.randint(0, M - 1, (N,), generator=g, device="cuda")[q]) % M
            b[q, j] = _uniform(g, 1.0, 4.0, N)[q]
            A[q, k] = -A[q, j]
            b[q, k] = -(b[q, j] + _uniform(g, 0.5, 1.0, N)[q])
        q = torch.nonzero((u >= 0.225) & (u < 0.25)).flatten()
        j = torch.randint(0, K, (N,), generator=g, device="cuda")[q]
        A[q, :, j] = _uniform(g, -1.0, 0.0, N, M)[q]
        c[q, j] = _uniform(g, 0.5, 1.0, N)[q]
    return m, n, a_off, b_off, c_off, A.reshape(-1).contiguous(), b.reshape(-1).contiguous(), c.reshape(-1).contiguous()


class _Batch:
    """One batch handle and the device arrays its results go to."""

    def __init__(self, data, precision):
        m, n, a_off, b_off, c_off, A, b, c = data
        opts = lpb.lpb_default_opts(precision=_precision(precision))
        self.h = lpb.lp_batch_create(m, n, a_off, A, b_off, b, c_off, c, lpb.LPB_DEVICE, opts,
                                     torch.cuda.current_stream())
        N = len(m)
        self.out = _out(N, int(m.sum(dtype=np.int64)), int(n.sum(dtype=np.int64)), "cuda")

    def results(self):
        o = self.out
        lpb.lp_batch_results(self.h, o["status"], o["iters"], o["obj"], o["x"], o["y"], lpb.LPB_DEVICE)
        return o

    def __del__(self):
        if getattr(self, "h", None) is not None:
            lpb.lp_batch_destroy(self.h)


def _precision(name):
    return lpb.LP_PREC_FP64 if name == "fp64" else lpb.LP_PREC_FP32_REFINE


def _out(N, rows, cols, device):
    kw = {"device": device, "pin_memory": device == "cpu"}
    return {"status": torch.zeros(N, dtype=torch.int32, **kw), "iters": torch.zeros(N, dtype=torch.int32, **kw),
            "obj": torch.zeros(N, dtype=F64, **kw), "x": torch.zeros(cols, dtype=F64, **kw),
            "y": torch.zeros(rows, dtype=F64, **kw)}


# -- the warm start's network --

_TRAIN_LPS = 16384


def _params(case, seed):
    """He-uniform weights and zero biases in the library's layout, one flat FP32 array."""
    m, n = case["m"], case["n"]
    hidden = case.get("hidden", 512)
    rs = np.random.RandomState((int(seed) * 11 + 5) % (1 << 31))
    p = []
    for i, o in ((m + n, hidden), (hidden, hidden), (hidden, m)):
        p += [rs.uniform(-1, 1, (o, i)).astype(np.float32) * math.sqrt(6.0 / i), np.zeros(o, np.float32)]
    return p


def _features(data, m, n):
    return torch.cat([data[6].view(-1, m), data[7].view(-1, n)], 1).float()


def _scaling(x):
    mean, std = x.double().mean(0), x.double().std(0, unbiased=False)
    return mean.float(), (1.0 / std).float()


def _logits(p, x):
    h = torch.relu(x @ p[0].T + p[1])
    h = torch.relu(h @ p[2].T + p[3])
    return h @ p[4].T + p[5]


def _trained(case, seed):
    """Weights and scaling of a network trained (here by PyTorch, so that they do not depend on the
    library's own training) on LPs of the case's family: which rows are active at the optimum."""
    m, n, N = case["m"], case["n"], _TRAIN_LPS
    data = list(_batch(case, seed))
    g = _gen(seed + 1_000_003)
    b0 = data[6].view(-1, m).mean(0)
    data[0], data[1] = np.full(N, m, np.int32), np.full(N, n, np.int32)
    data[2], data[3], data[4] = np.zeros(N, np.int64), np.arange(N, dtype=np.int64) * m, np.arange(N, dtype=np.int64) * n
    data[6] = (b0 * (1.0 + 0.1 * torch.randn((N, m), generator=g, device="cuda", dtype=F64))).reshape(-1).contiguous()
    data[7] = _uniform(g, 0.0, 1.0, N * n)
    cold = _Batch(data, "fp64")
    lpb.lp_batch_solve(cold.h, torch.cuda.current_stream())
    y = (cold.results()["y"].view(N, m) > 0).float()
    x = _features(data, m, n)
    mean, inv = _scaling(x)
    x = (x - mean) * inv
    p = [torch.from_numpy(v).cuda().requires_grad_(True) for v in _params(case, seed)]
    opt = torch.optim.Adam(p, lr=2e-3)
    w = torch.full((), 4.0, device="cuda")
    for t in range(160):
        at = (t * 1024) % N
        loss = torch.nn.functional.binary_cross_entropy_with_logits(_logits(p, x[at:at + 1024]), y[at:at + 1024],
                                                                    pos_weight=w)
        opt.zero_grad()
        loss.backward()
        opt.step()
    return np.concatenate([v.detach().cpu().numpy().ravel() for v in p]), mean, inv


def prepare(case, seed):
    call = case["call"]
    if call == "hyperbox":
        g = _gen(seed)
        N, dim = case["num"], case["dim"]
        L = torch.randn((N, dim), generator=g, device="cuda", dtype=F64)
        L /= L.norm(dim=1, keepdim=True)
        shape = (N, dim) if case["per_lp"] else (dim,)
        lo = _uniform(g, -2.0, 0.0, *shape)
        hi = lo + _uniform(g, 0.5, 3.0, *shape)
        return {"call": call, "L": L, "lo": lo, "hi": hi, "per_lp": case["per_lp"],
                "obj": torch.empty(N, dtype=F64, device="cuda"),
                "x": torch.empty((N, dim), dtype=F64, device="cuda") if case["with_x"] else None}
    if call == "train":
        return _train_state(case, seed)
    data = _batch(case, seed)
    m, n, a_off, b_off, c_off, A, b, c = data
    opts = lpb.lpb_default_opts(precision=_precision(case["precision"]))
    N, rows, cols = case["num"], int(m.sum(dtype=np.int64)), int(n.sum(dtype=np.int64))
    if call == "host":
        pinned = [torch.empty(v.shape, dtype=F64, pin_memory=True).copy_(v) for v in (A, b, c)]
        return {"call": call, "sizes": (m, n), "off": (a_off, b_off, c_off), "data": pinned, "opts": opts,
                "out": _out(N, rows, cols, "cpu")}
    if call == "noalloc":
        return {"call": call, "shape": (N, case["m"], case["n"]), "data": (A, b, c), "opts": opts,
                "out": _out(N, rows, cols, "cuda")}
    state = {"call": call, "batch": _Batch(data, case["precision"])}
    if call == "warm":
        p, mean, inv = _trained(case, seed)
        net = lpb.Mlp(case["m"] + case["n"], 512, 512, case["m"], max_batch=1024)
        net.set_params(p)
        net.set_scaling(mean.cpu().numpy(), inv.cpu().numpy())
        state["net"] = net
    return state


def _train_data(case, seed):
    """Scaled-down training data: features of the shared-matrix family, targets with
    the density of its active rows (the network's cost does not depend on them)."""
    g = _gen(seed)
    m, n, B = case["m"], case["n"], case["batch"] * case["steps"]
    b0 = _uniform(g, 1.0, 100.0, m)
    b = b0 * (1.0 + 0.1 * torch.randn((B, m), generator=g, device="cuda", dtype=F64))
    c = _uniform(g, 0.0, 1.0, B, n)
    score = b / b0 + 0.02 * (c.mean(1, keepdim=True) - 0.5)
    rank = (b0.argsort().argsort() < max(1, m // 18))
    y = ((score < 1.05) & rank).float()
    return torch.cat([b, c], 1).float(), y.contiguous()


def _train_state(case, seed):
    x, y = _train_data(case, seed)
    mean, inv = _scaling(x)
    net = lpb.Mlp(case["m"] + case["n"], case["hidden"], case["hidden"], case["m"], max_batch=case["batch"])
    net.set_params(np.concatenate([v.ravel() for v in _params(case, seed)]))
    net.set_scaling(mean.cpu().numpy(), inv.cpu().numpy())
    return {"call": "train", "net": net, "x": x, "y": y, "batch": case["batch"], "steps": case["steps"]}


_LR, _POS_WEIGHT = 1e-3, 4.0


def run(state):
    call = state["call"]
    stream = torch.cuda.current_stream()
    if call == "hyperbox":
        lpb.lp_hyperbox_solve(state["L"], state["lo"], state["hi"], state["obj"], state["x"], state["per_lp"],
                              lpb.LPB_DEVICE, stream)
        return {"obj": state["obj"]} if state["x"] is None else {"obj": state["obj"], "x": state["x"]}
    if call == "train":
        net, B, loss = state["net"], state["batch"], None
        for t in range(state["steps"]):
            at = t * B
            loss = net.train_step(state["x"][at:at + B], state["y"][at:at + B], _LR, _POS_WEIGHT,
                                  want_loss=t == state["steps"] - 1, stream=stream)
        return {"params": net.get_params(), "loss": loss}
    if call == "host":
        (m, n), (ao, bo, co), (A, b, c), o = state["sizes"], state["off"], state["data"], state["out"]
        lpb.lp_solve_host(m, n, ao, A, bo, b, co, c, o["status"], o["iters"], o["obj"], o["x"], o["y"], state["opts"])
        return o
    if call == "noalloc":
        (N, m, n), (A, b, c), o = state["shape"], state["data"], state["out"]
        code = lpb.lp_solve_uniform_noalloc(N, m, n, A, b, c, o["status"], o["iters"], o["obj"], o["x"], o["y"],
                                            state["opts"], stream)
        if code != lpb.LPB_OK:
            raise RuntimeError(lpb.strerror(code))
        return o
    batch = state["batch"]
    if call == "warm":
        lpb.lp_batch_solve_warm(batch.h, state["net"], 0.2, stream)
    else:
        lpb.lp_batch_solve(batch.h, stream)
    return batch.results()


def work(case):
    call = case["call"]
    if call == "hyperbox":
        N, d = case["num"], case["dim"]
        box = 2 * d * (N if case["per_lp"] else 1)
        return {"bytes": 8 * (N * d + box + N + (N * d if case["with_x"] else 0)), "flops": 2 * N * d}
    if call == "train":
        m, n, h, B, S = case["m"], case["n"], case["hidden"], case["batch"], case["steps"]
        weights = (m + n) * h + h * h + h * m
        # the three layers' products, forward and both gradients (the first layer's input has none)
        return {"bytes": 4 * (S * B * (2 * m + n) + 2 * weights), "flops": 2 * B * S * (3 * weights - (m + n) * h)}
    # The pivots that an LP takes are not known beforehand: its data read once, its results written once, and the
    # product A x that any check of an answer takes.
    N, M, K = case["num"], case["m"], case["n"]
    if case["family"] == "uneven":
        lo = case["lo"]
        M = (M - lo) / math.log(M / lo)  # mean of a log-uniform size
        K = (K - lo) / math.log(K / lo)
    shared_a, shared_b = case["family"] in ("support", "shared"), case["family"] == "support"
    inputs = M * K * (1 if shared_a else N) + M * (1 if shared_b else N) + K * N
    return {"bytes": 8 * inputs + N * (16 + 8 * (M + K)), "flops": 2 * M * K * N}


# ---------------------------------------------------------------------------
# The same results in 64 bits, in plain PyTorch
# ---------------------------------------------------------------------------

def exact(case, seed):
    call = case["call"]
    if call == "hyperbox":
        s = prepare(case, seed)
        h = torch.where(s["L"] < 0, s["lo"], s["hi"])
        obj = (s["L"] * h).sum(1)
        return {"obj": obj, "x": h} if case["with_x"] else {"obj": obj}
    if call == "train":
        return _exact_train(case, seed)
    if case["family"] == "mixed_sign" and case["precision"] == "mixed":
        # about half of these LPs are unbounded or infeasible: what is reported for
        # them is the last basis of an FP32 run, which 64 bits do not give
        return None
    m, n, a_off, b_off, c_off, A, b, c = _batch(case, seed)
    N = case["num"]
    obj = torch.zeros(N, dtype=F64, device="cuda")
    x = torch.zeros(int(n.sum(dtype=np.int64)), dtype=F64, device="cuda")
    y = torch.zeros(int(m.sum(dtype=np.int64)), dtype=F64, device="cuda")
    x_off, y_off = _offsets(n), _offsets(m)
    by = np.lexsort((n, m // 16)) if case["family"] == "uneven" else np.arange(N)
    at = 0
    while at < N:
        # LPs of like sizes together, padded with empty rows and columns, within 4 GB
        most = int(n[by[at:at + 4096]].max()) * int(m[by[at:at + 4096]].max()) if at < N else 1
        cnt = max(1, min(N - at, int(5e8 / (most + 1) / (2 if case["family"] == "mixed_sign" else 1))))
        idx = by[at:at + cnt]
        at += cnt
        _solve_block(idx, m, n, a_off, b_off, c_off, A, b, c, obj, x, y, x_off, y_off)
    return {"status": None, "iters": None, "obj": obj, "x": x, "y": y}


def _gather(flat, off, rows, cols, R, C):
    """[L, R, C] blocks from the flat array (row-major rows x cols each), zeros beyond."""
    dev = flat.device
    off, rows, cols = (torch.from_numpy(np.asarray(v, np.int64)).to(dev) for v in (off, rows, cols))
    r, q = torch.arange(R, device=dev), torch.arange(C, device=dev)
    inside = (r[None, :, None] < rows[:, None, None]) & (q[None, None, :] < cols[:, None, None])
    at = off[:, None, None] + r[None, :, None] * cols[:, None, None] + q[None, None, :]
    return torch.where(inside, flat[torch.where(inside, at, torch.zeros_like(at))], 0.0)


def _solve_block(idx, m, n, a_off, b_off, c_off, A, b, c, obj, x, y, x_off, y_off):
    """The two-phase simplex method with Dantzig's rule on a block of LPs at once (condensed tableau:
    column 0 the right-hand side, one column per non-basic variable)."""
    mi, ni = m[idx], n[idx]
    R, C = int(mi.max()), int(ni.max())
    L = len(idx)
    dev = A.device
    T0 = _gather(A, a_off[idx], mi, ni, R, C)
    B0 = _gather(b, b_off[idx], mi, np.ones_like(mi), R, 1)[:, :, 0]
    C0 = _gather(c, c_off[idx], np.ones_like(ni), ni, 1, C)[:, 0]
    rows, cols = torch.from_numpy(mi.astype(np.int64)).to(dev), torch.from_numpy(ni.astype(np.int64)).to(dev)
    negrow = B0 < 0
    k = int(negrow.sum(1).max())
    # rows 0..R-1 constraints, R objective, R+1 auxiliary objective of phase I
    T = torch.zeros((L, R + 2, 1 + C + k), dtype=F64, device=dev)
    T[:, :R, 1:1 + C] = T0
    T[:, :R, 0] = B0
    T[:, R, 1:1 + C] = -C0
    art, slack = C + R, C  # variables: structural j, slack C + i, artificial C + R + t
    rowvar = (slack + torch.arange(R, device=dev)).repeat(L, 1)
    colvar = torch.full((L, 1 + C + k), -1, dtype=torch.long, device=dev)
    colvar[:, 1:1 + C] = torch.arange(C, device=dev)
    if k:
        lp, i = torch.nonzero(negrow, as_tuple=True)
        t = (negrow.long().cumsum(1) - 1)[lp, i]
        T[lp, i] = -T[lp, i]
        rowvar[lp, i] = art + t
        T[lp, i, 1 + C + t] = -1.0
        colvar[lp, 1 + C + t] = slack + i
        w = -(T[:, :R] * negrow[:, :, None]).sum(1)
        T[:, R + 1] = w
    phase1 = negrow.any(1)
    bmax = B0.abs().amax(1).clamp(min=1.0)
    ids = torch.arange(L, device=dev)
    done_T = T.clone()
    done_rv, done_cv, done_y = rowvar.clone(), colvar.clone(), torch.full((L,), R, device=dev)
    live_row = torch.arange(R, device=dev)[None] < rows[:, None]
    live_col0 = torch.arange(C, device=dev)[None] < cols[:, None]
    live = torch.cat([torch.zeros((L, 1), dtype=torch.bool, device=dev), live_col0,
                      colvar[:, 1 + C:] >= 0], 1)

    def finish(mask, yrow):
        q = ids[mask]
        done_T[q], done_rv[q], done_cv[q], done_y[q] = T[mask], rowvar[mask], colvar[mask], yrow

    def pivot(sel, l, e):
        """Pivot the LPs `sel` (indices into the block's live LPs) on row l, column e."""
        q = torch.arange(len(sel), device=dev)
        sub = T[sel]
        col = sub[q, :, e].clone()
        pe = col[q, l]
        row = sub[q, l] / pe[:, None]
        row[q, e] = 1.0 / pe
        sub[q, :, e] = 0.0
        sub -= col[:, :, None] * row[:, None, :]
        sub[q, l] = row
        T[sel] = sub
        out = rowvar[sel, l].clone()
        rowvar[sel, l] = colvar[sel, e]
        colvar[sel, e] = out
        live[sel, e] = out < art  # an artificial never comes back

    inf = float("inf")
    for _ in range(50 * (R + C)):
        if not len(ids):
            break
        every = torch.arange(len(ids), device=dev)
        orow = T[every, torch.where(phase1, R + 1, R)]
        d = torch.where(live, orow, inf)
        dmin, e = d.min(1)
        stop = dmin >= -1e-9
        end1 = stop & phase1
        if end1.any():
            infeasible = end1 & (-T[:, R + 1, 0] > 1e-9 * bmax)
            go = end1 & ~infeasible
            for i in range(R):  # artificials still basic at 0 leave on the lowest usable column
                at = torch.nonzero(go & (rowvar[:, i] >= art)).flatten()
                if not len(at):
                    continue
                ok = live[at] & (T[at, i].abs() > 1e-9)
                label = torch.where(ok, colvar[at], 1 << 40)
                best, col = label.min(1)
                at, col = at[best < (1 << 40)], col[best < (1 << 40)]
                if len(at):
                    T[at, R + 1] = 0.0
                    pivot(at, torch.full_like(at, i), col)
            phase1 = phase1 & ~go
        else:
            infeasible = torch.zeros_like(stop)
        optimal = stop & ~phase1 & ~end1
        colE = T[every, :R, e]
        able = (colE > 1e-9) & live_row
        ratio = torch.where(able, T[:, :R, 0] / torch.where(able, colE, 1.0), inf)
        rmin, l = ratio.min(1)
        unbounded = ~stop & (rmin == inf)
        over = optimal | unbounded | infeasible
        if infeasible.any():
            finish(infeasible, R + 1)
        if (optimal | unbounded).any():
            finish(optimal | unbounded, R)
        move = torch.nonzero(~stop & ~over).flatten()
        if len(move):
            pivot(move, l[move], e[move])
        if over.any():
            keep = ~over
            ids, T, rowvar, colvar, live = ids[keep], T[keep], rowvar[keep], colvar[keep], live[keep]
            phase1, bmax, live_row = phase1[keep], bmax[keep], live_row[keep]

    xs = torch.zeros((L, art + k + 1), dtype=F64, device=dev)
    xs.scatter_(1, done_rv, done_T[:, :R, 0])
    ys = torch.zeros((L, art + k + 1), dtype=F64, device=dev)
    ys.scatter_(1, torch.where(done_cv >= 0, done_cv, art + k), done_T[torch.arange(L, device=dev), done_y])
    lo = torch.from_numpy(idx.astype(np.int64)).to(dev)
    obj[lo] = done_T[:, R, 0]
    for dst, off, val, cnt, W in ((x, x_off, xs[:, :C], cols, C), (y, y_off, ys[:, slack:slack + R], rows, R)):
        q = torch.arange(W, device=dev)
        ok = q[None] < cnt[:, None]
        at = torch.from_numpy(off[idx]).to(dev)[:, None] + q[None]
        dst[at[ok]] = val[ok]


def _exact_train(case, seed):
    x, y = _train_data(case, seed)
    mean, inv = _scaling(x)
    x = ((x.double() - mean.double()) * inv.double())
    y = y.double()
    p = [torch.from_numpy(v).cuda().double().requires_grad_(True) for v in _params(case, seed)]
    mom, var = [torch.zeros_like(v) for v in p], [torch.zeros_like(v) for v in p]
    B, loss = case["batch"], None
    w = torch.full((), _POS_WEIGHT, device="cuda", dtype=F64)
    for t in range(case["steps"]):
        at = t * B
        loss = torch.nn.functional.binary_cross_entropy_with_logits(_logits(p, x[at:at + B]), y[at:at + B], pos_weight=w)
        grads = torch.autograd.grad(loss, p)
        with torch.no_grad():
            for v, g, a, q in zip(p, grads, mom, var):
                a.mul_(0.9).add_(0.1 * g)
                q.mul_(0.999).add_(0.001 * g * g)
                v -= _LR * (a / (1 - 0.9 ** (t + 1))) / ((q / (1 - 0.999 ** (t + 1))).sqrt() + 1e-8)
    return {"params": np.concatenate([v.detach().cpu().numpy().ravel() for v in p]), "loss": float(loss)}
