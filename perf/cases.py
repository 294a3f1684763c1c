"""The work a user of this library has it do, as cases to be measured.

Every case goes through the public entry points of ``l1line`` the way a
program that calls them in a loop does: inputs, workspace, output buffers and
the network are in hand before the call, and one call is one pass.  Sizes and
distributions are those of the library's own workloads (``datagen``) and of the
ranges its tests cover.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2402_16712_gb300 import datagen, l1line, proposer

F32, F64 = "float32", "float64"


# ---------------------------------------------------------------------------
# The listed cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # One fit of a small sample, the call inside someone's cross-validation
        # loop: latency and launches are all of it.
        {"name": "fit_small_f64", "kind": "fit", "dtype": F64, "n": 200, "m": 20, "lams": 1,
         "lam": 0.1, "nnz": 4, "noise": 0.05, "frac": 0.10, "std": 5.0},
        # The paper's size, one penalty: the library's headline workload.
        {"name": "fit_paper_f32", "kind": "fit", "dtype": F32, "n": 2000, "m": 2000, "lams": 1,
         "lam": 0.5, "nnz": 20, "noise": 0.1, "frac": 0.05, "std": 10.0},
        # The same in double, for users whose data is double.
        {"name": "fit_paper_f64", "kind": "fit", "dtype": F64, "n": 2000, "m": 2000, "lams": 1,
         "lam": 0.5, "nnz": 20, "noise": 0.1, "frac": 0.05, "std": 10.0},
        # A grid of 32 penalties over one matrix: choosing lambda.
        {"name": "fit_lambdas_f32", "kind": "fit", "dtype": F32, "n": 1000, "m": 500, "lams": 32,
         "lam": 1.0, "nnz": 10, "noise": 0.1, "frac": 0.10, "std": 10.0},
        # Every v, residual and objective of a long matrix of odd sizes (what
        # labels the proposer's training set, and what a user inspects).
        {"name": "scan_long_f32", "kind": "scan", "dtype": F32, "n": 4999, "m": 1001, "lams": 1,
         "lam": 0.2, "nnz": 60, "noise": 0.1, "frac": 0.10, "std": 10.0},
        # More rows than shared memory holds, few coordinates: the kernel that
        # streams its columns.
        {"name": "fit_tall_f32", "kind": "fit", "dtype": F32, "n": 1000000, "m": 16, "lams": 1,
         "lam": 0.5, "nnz": 4, "noise": 0.1, "frac": 0.05, "std": 10.0},
        # 256 independent matrices of uneven size in one call.
        {"name": "batch_uneven_f32", "kind": "batch", "dtype": F32, "count": 256, "n_lo": 100,
         "n_hi": 5000, "m_lo": 10, "m_hi": 500, "lams": 1, "model": "planted", "shape_seed": 0},
        # A simulation study: 30 small double matrices, 8 penalties each.
        {"name": "batch_study_f64", "kind": "batch", "dtype": F64, "count": 30, "n_lo": 100,
         "n_hi": 100, "m_lo": 100, "m_hi": 100, "lams": 8, "model": "study", "shape_seed": 0},
        # The learned path: network-proposed candidates, fitted exactly.
        {"name": "proposed_f32", "kind": "proposed", "dtype": F32, "n": 5000, "m": 1000, "K": 32,
         "lam": 0.2, "nnz": 50, "noise": 0.1, "frac": 0.10, "std": 10.0},
        # One training step of that network on 16 instances' candidates.
        {"name": "train_step", "kind": "train", "inst": 16, "m_lo": 100, "m_hi": 1000,
         "shape_seed": 0},
        # Every pair's penalty path (Algorithm 2), into buffers with room for
        # `room` entries per pair.
        {"name": "paths_f32", "kind": "paths", "dtype": F32, "n": 2000, "m": 400, "room": 90,
         "nnz": 10, "noise": 0.1, "frac": 0.05, "std": 10.0},
        # The whole solution path over all penalties (Algorithms 2 and 3).
        {"name": "solution_f32", "kind": "solution", "dtype": F32, "n": 1000, "m": 500,
         "room": 70, "nnz": 10, "noise": 0.1, "frac": 0.10, "std": 10.0},
    ]


# ---------------------------------------------------------------------------
# Drawn cases: the same kinds over their ranges
# ---------------------------------------------------------------------------
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _model(rng, m):
    return {"nnz": rng.randint(1, max(1, m // 10)), "noise": rng.choice([0.05, 0.1]),
            "frac": round(rng.uniform(0.0, 0.2), 3), "std": rng.choice([5.0, 10.0])}


def draw(rng):
    kind = rng.choice(["fit", "fit", "fit", "scan", "lambdas", "tall", "batch", "study",
                       "proposed", "train", "paths", "solution"])
    dtype = rng.choice([F32, F32, F64])
    lam = round(10.0 ** rng.uniform(-2.0, 1.0), 4)
    if kind in ("fit", "scan"):
        n = _log(rng, 60, 12000)
        m = _log(rng, 10, 2000)
        while n * m * m > 8.0e9:  # at most the listed paper size
            n, m = _log(rng, 60, 12000), _log(rng, 10, 2000)
        return {"kind": kind, "dtype": dtype, "n": n, "m": m, "lams": 1, "lam": lam,
                **_model(rng, m)}
    if kind == "lambdas":
        n, m = _log(rng, 100, 3000), _log(rng, 20, 500)
        return {"kind": "fit", "dtype": dtype, "n": n, "m": m, "lams": rng.randint(2, 64),
                "lam": 1.0, **_model(rng, m)}
    if kind == "tall":
        n, m = _log(rng, 21000, 1000000), rng.randint(2, 16)
        return {"kind": "fit", "dtype": dtype, "n": n, "m": m, "lams": 1, "lam": lam,
                **_model(rng, m)}
    if kind == "batch":
        return {"kind": "batch", "dtype": dtype, "count": rng.randint(8, 128), "n_lo": 100,
                "n_hi": _log(rng, 300, 5000), "m_lo": 10, "m_hi": _log(rng, 30, 300),
                "lams": rng.choice([1, 1, 4]), "model": "planted",
                "shape_seed": rng.randint(1, 10 ** 6)}
    if kind == "study":
        s = rng.randint(60, 150)
        return {"kind": "batch", "dtype": F64, "count": rng.randint(10, 40), "n_lo": s, "n_hi": s,
                "m_lo": s, "m_hi": s, "lams": rng.randint(1, 12), "model": "study",
                "shape_seed": rng.randint(1, 10 ** 6)}
    if kind == "proposed":
        n, m = _log(rng, 500, 5000), _log(rng, 100, 1000)
        return {"kind": "proposed", "dtype": dtype, "n": n, "m": m,
                "K": rng.choice([k for k in (16, 32, 64, 128) if k <= m]), "lam": 0.2,
                **_model(rng, m)}
    if kind == "train":
        return {"kind": "train", "inst": rng.randint(4, 64), "m_lo": 100,
                "m_hi": _log(rng, 150, 1000), "shape_seed": rng.randint(1, 10 ** 6)}
    n, m = _log(rng, 100, 2000), _log(rng, 20, 300)
    room = min(n + 1, 8 + int(n * (0.1 + 2.0 / math.sqrt(n))))
    return {"kind": kind, "dtype": dtype, "n": n, "m": m, "room": room, **_model(rng, m)}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _matrix(case, seed, n=None, m=None):
    """The planted sparse line of the library's workloads, drawn on the GPU."""
    X, _, _ = datagen.planted_torch(
        datagen.Planted(n or case["n"], m or case["m"], case["nnz"], case["noise"], case["frac"],
                        case["std"], seed, case["dtype"]), "cuda")
    return X


def _lams(case):
    if case.get("lams", 1) == 1:
        return np.array([case.get("lam", 0.2)])
    return np.logspace(-3, 1, case["lams"])


def _shapes(case):
    """Sizes of a batch's matrices: part of the case, the same for every seed."""
    rng = np.random.default_rng(case["shape_seed"])
    out = []
    for _ in range(case["count"]):
        n = int(rng.integers(case["n_lo"], case["n_hi"] + 1))
        m = int(rng.integers(case["m_lo"], case["m_hi"] + 1))
        out.append((n, m, int(rng.integers(1, max(1, m // 10) + 1)), float(rng.uniform(0, 0.2))))
    return out


def _batch(case, seed):
    Xs = []
    for b, (n, m, nnz, frac) in enumerate(_shapes(case)):
        s = seed * 100003 + b + 1
        if case["model"] == "study":
            X = torch.from_numpy(datagen.comparison(s, 1 + b % 6, n, m, case["dtype"])[0]).cuda()
        else:
            X = datagen.planted_torch(
                datagen.Planted(n, m, nnz, 0.1, frac, 10.0, s, case["dtype"]), "cuda")[0]
        Xs.append(X)
    return Xs, [_lams(case)] * len(Xs)


def _train(case, seed):
    """Standardised features and targets of a step's candidates, the network
    and Adam's moments as they stand some way into training."""
    shapes = np.random.default_rng(case["shape_seed"])
    ms = shapes.integers(case["m_lo"], case["m_hi"] + 1, size=case["inst"])
    off = np.concatenate([[0], np.cumsum(ms)]).astype(np.int64)
    N = int(off[-1])
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def rnd(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32)

    feat = rnd(N, l1line.MLP_FEATURES)
    # the targets follow the features, loosely: -(z - z_min) / (T span)
    tgt = (-4.0 * (feat[:, 3] - 0.3 * feat[:, 1] + 0.2 * rnd(N) + 3.0).abs()).contiguous()
    rows = torch.randperm(N, generator=g, device="cuda").to(torch.int32)
    theta = torch.from_numpy(proposer.init_theta(seed)).cuda()
    m1 = 1e-3 * rnd(l1line.MLP_PARAMS)
    m2 = (1e-3 * rnd(l1line.MLP_PARAMS)) ** 2 + 1e-7
    return {"feat": feat, "tgt": tgt, "rows": rows, "theta": theta, "m1": m1, "m2": m2,
            "off": torch.from_numpy(off).cuda(), "step": 100, "N": N}


def _path_buffers(X, entries, solution):
    """Outputs and workspaces of the penalty-path calls, with room for `entries`
    breakpoints (zero where a pair does not fill its room)."""
    n, m = X.shape

    def zeros(shape, dtype):
        return torch.zeros(shape, dtype=dtype, device="cuda")

    st = {"ws": l1line.path_workspace(X.dtype, n, m), "entries": entries,
          "off": zeros(m * m + 1, torch.int64), "lam": zeros(entries, torch.float64),
          "v": zeros(entries, X.dtype), "len": zeros(m * m, torch.int32)}
    if solution:
        cap = 500 + int(0.06 * n * m)
        need = l1line.load().l1line_solution_path_workspace_bytes(m, entries)
        st.update(res=zeros(entries, torch.float64), sws=l1line.Workspace(need), cap=cap,
                  start=zeros(cap, torch.float64), jhat=zeros(cap, torch.int32),
                  icpt=zeros(cap, torch.float64), slope=zeros(cap, torch.float64),
                  sv=zeros((cap, m), X.dtype), count=zeros(1, torch.int64))
    return st


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        Xs, lams = _batch(case, seed)
        return {"kind": kind, "batch": l1line.Batched(Xs, lams)}
    if kind == "train":
        st = _train(case, seed)
        N = st["N"]
        st.update(kind=kind, mlp=l1line.mlp_pack(st["theta"]),
                  score=torch.empty(N, device="cuda"), ds=torch.empty(N, device="cuda"),
                  loss=torch.empty(case["inst"], device="cuda"),
                  grad=torch.empty(l1line.MLP_PARAMS, device="cuda"),
                  ws=l1line.MlpWorkspace(N))
        return st
    X = _matrix(case, seed)
    n, m = X.shape
    st = {"kind": kind, "X": X, "lams": _lams(case)}
    nl = len(st["lams"])
    if kind in ("paths", "solution"):
        st.update(_path_buffers(X, m * m * case["room"], kind == "solution"))
    elif kind == "scan":
        st["ws"] = l1line.Workspace.for_shape(X.dtype, n, m, nl)
        st["out"] = (torch.empty((nl, m, m), dtype=X.dtype, device="cuda"),
                     torch.empty((nl, m, m), dtype=torch.float64, device="cuda"),
                     torch.empty((nl, m), dtype=torch.float64, device="cuda"))
    elif kind in ("fit", "proposed"):
        st["out"] = (torch.empty((nl, m), dtype=X.dtype, device="cuda"),
                     torch.empty(nl, dtype=torch.float64, device="cuda"),
                     torch.empty(nl, dtype=torch.int32, device="cuda"))
        if kind == "fit":
            st["ws"] = l1line.Workspace.for_shape(X.dtype, n, m, nl)
        else:
            st["ws"] = l1line.proposed_workspace(X.dtype, n, m, nl)
            st["mlp"] = proposer.network()
            st["K"] = case["K"]
            st["idx"] = torch.empty(case["K"], dtype=torch.int32, device="cuda")
    return st


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(st):
    kind = st["kind"]
    if kind == "fit":
        v, obj, js, _ = l1line.fit(st["X"], st["lams"], workspace=st["ws"], out=st["out"])
        return {"v": v, "obj": obj, "jstar": js}
    if kind == "scan":
        v, s, z, _ = l1line.scan(st["X"], st["lams"], workspace=st["ws"], out=st["out"])
        return {"v": v, "s": s, "z": z}
    if kind == "batch":
        b = st["batch"]
        b.run()
        return {"v": b.out_v, "obj": b.out_obj, "jstar": b.out_jstar}
    if kind == "proposed":
        v, obj, js, idx, _ = l1line.fit_proposed(st["X"], st["lams"], st["mlp"], st["K"],
                                                 workspace=st["ws"], out=st["out"], idx=st["idx"])
        return {"v": v, "obj": obj, "jstar": js, "idx": idx}
    if kind == "train":
        l1line.mlp_forward(st["feat"], st["mlp"], rows=st["rows"], out=st["score"])
        l1line.rank_loss(st["score"], st["tgt"], st["off"], rows=st["rows"], dscores=st["ds"],
                         loss=st["loss"])
        l1line.mlp_backward(st["feat"], st["mlp"], st["ds"], rows=st["rows"], grad=st["grad"],
                            workspace=st["ws"])
        l1line.adam_step(st["theta"], st["grad"], st["m1"], st["m2"], st["step"], 2e-3,
                         mlp=st["mlp"])
        st["step"] += 1
        return {"score": st["score"], "loss": st["loss"], "ds": st["ds"], "grad": st["grad"],
                "theta": st["theta"], "m1": st["m1"], "m2": st["m2"]}
    return _run_paths(st)


def _call(name, X, *args):
    """One call of the C ABI on the current stream."""
    f = getattr(l1line.load(), name + ("_f32" if X.dtype == torch.float32 else "_f64"))
    rc = f(*[a.data_ptr() if isinstance(a, torch.Tensor) else a for a in args],
           torch.cuda.current_stream().cuda_stream)
    if rc != l1line.OK:
        raise l1line.L1LineError(rc, name)


def _run_paths(st):
    X, ws, off = st["X"], st["ws"], st["off"]
    n, m = X.shape
    _call("l1line_path_count", X, X, n, m, off, ws.ptr, ws.nbytes)
    total = int(off[m * m])  # the program has to know that its buffers hold them
    if total > st["entries"]:
        raise RuntimeError(f"{total} entries, room for {st['entries']}")
    _call("l1line_path_write", X, X, n, m, off, st["lam"], st["v"], st.get("res"), st["len"],
          ws.ptr, ws.nbytes)
    out = {"offsets": off, "length": st["len"], "lam": st["lam"], "v": st["v"]}
    if "sws" not in st:
        return out
    sws = st["sws"]
    _call("l1line_solution_path", X, m, off, st["lam"], st["v"], st["res"], st["len"], total,
          st["start"], st["jhat"], st["icpt"], st["slope"], st["sv"], st["count"], st["cap"],
          sws.ptr, sws.nbytes)
    return {"start": st["start"], "jhat": st["jhat"], "intercept": st["icpt"],
            "slope": st["slope"], "v": st["sv"], "count": st["count"]}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: X once, the outputs once.  Flops: per (jhat, k) pair and row one
    multiply, one compare and one weight sum to rank the ratio, and a
    multiply-add and an absolute sum for the residual (6); the residual again
    for every further penalty (3)."""
    kind = case["kind"]
    es = 8 if case.get("dtype") == F64 else 4
    nl = case.get("lams", 1)
    if kind == "train":
        ms = np.random.default_rng(case["shape_seed"]).integers(case["m_lo"], case["m_hi"] + 1,
                                                                size=case["inst"])
        N, P = int(ms.sum()), l1line.MLP_PARAMS
        return {"bytes": N * (4 * 4 + 4 + 4 + 8) + P * 4 * 7, "flops": 6.0 * N * P}
    if kind == "batch":
        sh = _shapes(case)
        return {"bytes": sum(n * m * es + nl * (m * es + 12) for n, m, _, _ in sh),
                "flops": sum(float(n) * m * m * (6 + 3 * (nl - 1)) for n, m, _, _ in sh)}
    n, m = case["n"], case["m"]
    rows = float(n) * m * m
    if kind == "fit":
        return {"bytes": n * m * es + nl * (m * es + 12), "flops": rows * (6 + 3 * (nl - 1))}
    if kind == "scan":
        return {"bytes": n * m * es + nl * m * (m * (es + 8) + 8), "flops": 6 * rows}
    if kind == "proposed":
        sub = min(n, max(256, (n + 7) // 8))
        return {"bytes": n * m * es + m * es + 12 + 4 * case["K"],
                "flops": 6.0 * m * (m * sub + case["K"] * n)}
    # about 3% of a pair's rows lie between its median and 0
    entries = 0.03 * rows + m * m
    if kind == "paths":
        return {"bytes": n * m * es + entries * (8 + es) + m * m * 12.0, "flops": 8 * rows}
    return {"bytes": n * m * es + 2 * entries * (16 + es), "flops": 14 * rows}


# ---------------------------------------------------------------------------
# The same results in 64 bits by plain torch
# ---------------------------------------------------------------------------
def _exact_columns(X, lams, js, keep=False):
    """Algorithm 1's inner loops in double: objective z [nl, len(js)] of every
    jhat in js, and with keep also v and s [nl, len(js), m]."""
    X = X.to(torch.float64)
    n, m = X.shape
    XT = X.t().contiguous()
    nl = len(lams)
    z = torch.empty((nl, len(js)), dtype=torch.float64, device=X.device)
    V = torch.empty((nl, len(js), m), dtype=torch.float64, device=X.device) if keep else None
    S = torch.empty_like(V) if keep else None
    step = max(1, int(8e6 // (n * m)))
    for b0 in range(0, len(js), step):
        jb = js[b0:b0 + step]
        xj = XT[jb]
        w = xj.abs()
        r = XT[None] / xj[:, None, :]
        r = torch.where((w > 0)[:, None, :], r, math.inf)
        neg = torch.where(r <= 0, w[:, None, :], 0.0).sum(-1)
        rs, order = r.sort(dim=-1)
        cw = w[:, None, :].expand_as(r).gather(-1, order).cumsum(-1)
        tot = w.sum(-1)[:, None]
        diag = (torch.arange(len(jb), device=X.device), jb)
        for t, lam in enumerate(lams):
            lam = float(lam)
            # smallest ratio whose weight at or below it passes half the total
            half = (0.5 * (tot + lam))[..., None]
            below = torch.where(rs >= 0, cw + lam, cw) > half
            first = below.to(torch.uint8).argmax(-1, keepdim=True)
            v = rs.gather(-1, first)[..., 0]
            ok = below.gather(-1, first)[..., 0]
            v = torch.where(ok, v, 0.0)
            zero = (neg + lam > half[..., 0]) & (v > 0)  # the penalty point comes first
            v = torch.where(zero | ~torch.isfinite(v), 0.0, v)
            v[diag] = 1.0
            s = (XT[None] - v[..., None] * xj[:, None, :]).abs().sum(-1) + lam * v.abs()
            s[diag] = lam
            z[t, b0:b0 + len(jb)] = s.sum(-1)
            if keep:
                V[t, b0:b0 + len(jb)] = v
                S[t, b0:b0 + len(jb)] = s
    return z, V, S


def _exact_fit(X, lams, js=None):
    js = torch.arange(X.shape[1], device=X.device) if js is None else js
    z, _, _ = _exact_columns(X, lams, js)
    best = z.argmin(-1)
    v, obj = [], []
    for t in range(len(lams)):
        zt, V, _ = _exact_columns(X, lams[t:t + 1], js[best[t:t + 1]], keep=True)
        v.append(V[0, 0])
        obj.append(zt[0, 0])
    return torch.stack(v), torch.stack(obj), js[best].to(torch.int32)


def _exact_proposed(case, X, lams):
    n, m = X.shape
    A = X.to(torch.float64).abs()
    rho = torch.tensor(0.0, dtype=torch.float64, device=X.device)
    for j in range(m):
        rho = rho + A[:, j]
    R = min(n, max(256, (n + 7) // 8))
    rows = torch.sort(torch.sort(-rho.float(), stable=True).indices[:R]).values
    zr, _, _ = _exact_columns(X[rows], lams[:1], torch.arange(m, device=X.device))
    med = A.sort(dim=0).values[(n - 1) // 2]
    f = torch.stack([A.sum(0), (A * A).sum(0).sqrt(), med, zr[0]], 1).float().double()
    f = ((f - f.mean(0)) / f.std(0, correction=0)).float().double()
    s = _exact_forward(f, torch.from_numpy(proposer.load_theta()).cuda())[0]
    idx = torch.sort(torch.sort(-s, stable=True).indices[:case["K"]]).values
    return _exact_fit(X, lams, idx) + (idx.to(torch.int32),)


def _exact_forward(f, theta):
    H, F = 128, l1line.MLP_FEATURES
    w1, b1, w2, b2, w3, b3 = torch.split(theta, [H * F, H, H * H, H, H, 1])
    w1, w2, w3 = (x.half().double() for x in (w1, w2, w3))
    h1 = torch.relu(f @ w1.view(H, F).t() + b1.double())
    h2 = torch.relu(h1 @ w2.view(H, H).t() + b2.double())
    return h2 @ w3 + b3.double(), h1, h2, w2.view(H, H), w3


def _exact_train(st, inst):
    rows = st["rows"].long()
    f, tgt, off = st["feat"].double()[rows], st["tgt"].double()[rows], st["off"].tolist()
    s, h1, h2, w2, w3 = _exact_forward(f, st["theta"])
    ds, loss = torch.empty_like(s), []
    for b in range(inst):
        sl = slice(off[b], off[b + 1])
        q = torch.softmax(tgt[sl], 0)
        loss.append(torch.logsumexp(s[sl], 0) - (q * s[sl]).sum())
        ds[sl] = (torch.softmax(s[sl], 0) - q) / inst
    g2 = torch.where(h2 > 0, ds[:, None] * w3, 0.0)
    g1 = torch.where(h1 > 0, g2 @ w2, 0.0)
    grad = torch.cat([(g1.t() @ f).reshape(-1), g1.sum(0), (g2.t() @ h1).reshape(-1), g2.sum(0),
                      h2.t() @ ds, ds.sum()[None]])
    m1 = 0.9 * st["m1"].double() + 0.1 * grad
    m2 = 0.999 * st["m2"].double() + 0.001 * grad * grad
    c1, c2 = 1.0 / (1.0 - 0.9 ** st["step"]), 1.0 / (1.0 - 0.999 ** st["step"])
    theta = st["theta"].double() - 2e-3 * (m1 * c1) / ((m2 * c2).sqrt() + 1e-8)
    return {"score": s, "loss": torch.stack(loss), "ds": ds, "grad": grad, "theta": theta,
            "m1": m1, "m2": m2}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(_train(case, seed), case["inst"])
    if kind in ("paths", "solution"):
        # the breakpoints are those of ratios rounded to the input's precision:
        # in 64 bits their number, and so the layout, is another
        return None
    if kind == "batch":
        if sum(n * m * m for n, m, _, _ in _shapes(case)) > 6e9:
            return None  # minutes of sorting
        Xs, lams = _batch(case, seed)
        parts = [_exact_fit(X, l) for X, l in zip(Xs, lams)]
        return {"v": torch.cat([p[0].reshape(-1) for p in parts]),
                "obj": torch.cat([p[1] for p in parts]), "jstar": None}
    X, lams = _matrix(case, seed), _lams(case)
    if kind == "scan":
        z, v, s = _exact_columns(X, lams, torch.arange(X.shape[1], device="cuda"), keep=True)
        return {"v": v, "s": s, "z": z}
    if kind == "proposed":
        v, obj, js, idx = _exact_proposed(case, X, lams)
        return {"v": v, "obj": obj, "jstar": None, "idx": None}
    v, obj, js = _exact_fit(X, lams)
    return {"v": v, "obj": obj, "jstar": None}
