"""The library's work as its users have it done: one pass of each public path at the sizes it is
used at, from one small prediction to a whole learned factor build.

Point clouds, kernels, candidate counts and pick counts are those of `synthetic.PRESETS`, the
tests and the benchmark; N is scaled so that the host preparation stays short.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import synthetic
from paper_2307_11648_gb300 import gp, learned, pipeline, sic

DEV = "cuda"
PREC = {"fp64": sic.SIC_FP64, "fp32": sic.SIC_FP32_MIXED}
OPS = {"L": sic.SIC_OP_L, "LT": sic.SIC_OP_LT, "LLT": sic.SIC_OP_LLT}
MEAN_M = 23.3  # members per supernode at mmin 8, mmax 64 (mean over the preset's geometry)


def listed():
    return [
        # the headline path: one whole supernodal factor by the learned proposal
        dict(name="learned_step", kind="learned", n=1 << 18, dim=2, nu_x2=3, ell=0.02, nugget=1e-6, C=1024, top=256, k=64),
        # the plain reference build in double precision (the default precision), all 1024 candidates
        dict(name="plain_fp64", kind="groups", n=1 << 16, dim=2, nu_x2=3, ell=0.02, nugget=1e-6, C=1024, k=64, prec="fp64"),
        # one column at a time in three dimensions, mixed precision (preset cfg2)
        dict(name="columns_fp32", kind="columns", n=1 << 16, dim=3, nu_x2=5, ell=0.05, nugget=1e-6, C=512, k=32, prec="fp32"),
        # a small double-precision factor (preset cfg1)
        dict(name="columns_fp64", kind="columns", n=1 << 12, dim=2, nu_x2=3, ell=0.1, nugget=1e-8, C=256, k=16, prec="fp64"),
        # nonadjacent groups: partial selection and its fill
        dict(name="partial_fp32", kind="partial", n=1 << 16, dim=2, nu_x2=3, ell=0.02, nugget=1e-6, C=256, k=64, prec="fp32"),
        # a global nonzero budget on an inhomogeneous cloud, decreases from the FP64 side state
        dict(name="budget", kind="budget", n=1 << 16, dim=2, nu_x2=3, ell=0.02, nugget=1e-6, C=256, k=64, share=0.5),
        # new kernel parameters on a fixed pattern (a step of a likelihood fit): nnz scan and fill
        dict(name="refill", kind="refill", n=1 << 17, dim=2, nu_x2=3, ell=0.02, nugget=1e-6, k=64),
        # the preconditioner applied to a block of right-hand sides
        dict(name="apply_llt", kind="apply", n=1 << 17, dim=2, nu_x2=3, ell=0.02, nugget=1e-6, k=64, op="LLT", nrhs=8),
        # the dense kernel matrix applied on the fly (what an iteration of the solver spends its time on)
        dict(name="matvec_fp32", kind="matvec", n=50001, dim=2, nu_x2=3, ell=0.02, nugget=1e-6, prec="fp32", nrhs=8),
        # a few predictions by directed regression, host arrays in (the smallest call)
        dict(name="predict", kind="predict", n=4096, targets=37, dim=2, nu_x2=3, ell=0.1, nugget=1e-2, C=128, k=32),
        # conditional selection of one target among all training points
        dict(name="single_fp64", kind="single", n=1 << 16, dim=3, nu_x2=5, ell=0.2, nugget=1e-6, k=64, prec="fp64"),
        # one training step of the proposal network at the trainer's batch
        dict(name="train_step", kind="train", batch=65536),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["learned", "groups", "columns", "partial", "budget", "refill", "apply", "matvec", "predict",
                       "single", "train"])
    if kind == "train":
        return dict(kind=kind, batch=_log(rng, 1000, 65536))
    dim = rng.choice([2, 2, 3])
    c = dict(kind=kind, dim=dim, nu_x2=rng.choice([1, 3, 5]), ell=round(rng.uniform(0.02, 0.2), 4),
             nugget=rng.choice([1e-6, 1e-4, 1e-2]))
    if kind == "learned":
        c.update(n=_log(rng, 1 << 12, 1 << 17), C=_log(rng, 300, 1024), top=rng.choice([128, 256]), k=rng.randint(16, 64))
    elif kind == "groups":
        c.update(n=_log(rng, 1 << 11, 1 << 15), C=_log(rng, 128, 1024), k=rng.randint(16, 64),
                 prec=rng.choice(["fp64", "fp64", "fp32"]))
    elif kind == "columns":
        prec = rng.choice(["fp64", "fp32"])
        k = rng.randint(4, 64)
        top = (256 if k > 32 else 512) if prec == "fp64" else (512 if k > 32 else 1024)
        c.update(n=_log(rng, 1 << 10, 1 << (14 if prec == "fp64" else 16)), C=_log(rng, 64, top), k=k, prec=prec)
    elif kind == "partial":
        prec = rng.choice(["fp64", "fp32", "fp32"])
        c.update(n=_log(rng, 1 << 11, 1 << (14 if prec == "fp64" else 16)), C=_log(rng, 64, 128 if prec == "fp64" else 256),
                 k=rng.randint(16, 64), prec=prec)
    elif kind == "budget":
        c.update(n=_log(rng, 1 << 11, 1 << 16), C=_log(rng, 128, 256), k=rng.randint(16, 64), share=round(rng.uniform(0.2, 0.9), 3))
    elif kind == "refill":
        c.update(n=_log(rng, 1 << 11, 1 << 17), k=rng.randint(8, 96))
    elif kind == "apply":
        c.update(n=_log(rng, 1 << 11, 1 << 17), k=rng.randint(8, 64), op=rng.choice(["L", "LT", "LLT"]), nrhs=rng.randint(1, 8))
    elif kind == "matvec":
        prec = rng.choice(["fp64", "fp32", "fp32"])
        c.update(n=_log(rng, 1 << 10, 1 << (13 if prec == "fp64" else 15)), prec=prec, nrhs=rng.randint(1, 8))
    elif kind == "predict":
        c.update(n=_log(rng, 1 << 10, 1 << 16), targets=_log(rng, 1, 4096), C=_log(rng, 64, 256), k=rng.randint(8, 48))
    else:
        c.update(n=_log(rng, 1 << 8, 1 << 16), k=rng.randint(8, 64), prec=rng.choice(["fp64", "fp32"]))
    return c


# ------------------------------------------------------------------ inputs --

def _kernel(c):
    return sic.kernel(c["dim"], c["nu_x2"], c["ell"], 1.0, c["nugget"])


def _params(seed):
    """Network weights: the trainer's initial ones plus one hidden channel that falls with a candidate's
    relative distance to its nearest member, the main thing a trained network has learned."""
    p = learned.init_params(seed)
    p[0:17664] *= np.float32(0.3)
    p[2 * 128 + 0] = -4.0   # W1: feature 2 (relative distance) -> channel 0
    p[8 * 128 + 0] = 4.0    # b1
    p[1152 + 0] = 1.0       # W2: channel 0 -> channel 0
    p[17664 + 0] = 2.0      # w3
    return p


def _nearest_picks(hp):
    """The first k candidates (nearest first) of every unit as its picks."""
    U, k = hp.n_units, hp.k
    cnt = np.minimum(np.diff(hp.cand_ptr), k).astype(np.int32)
    sel = np.full((U, k), -1, np.int32)
    at = np.arange(k)[None, :] < cnt[:, None]
    sel[at] = hp.cand_idx[(hp.cand_ptr[:-1, None] + np.arange(k)[None, :])[at]]
    return sel, cnt


def _caps(c):
    """Bounds on the supernodes and the nonzeros at any seed (the grouping gives 15 or more members on average)."""
    return c["n"] // 12 + 16, c["n"] * (c["k"] + 32)


def _room(s, c, names):
    """Gives the builder's per-unit buffers their room for any seed's grouping; s["room"] has them whole, zero
    beyond what this grouping fills."""
    b, G = s["b"], _caps(c)[0]
    b = getattr(b, "fb", b)
    s["room"] = {}
    shared = getattr(b, "local_count", None) is b.sel_count  # without a budget the two counts are one buffer
    for name in names:
        x = getattr(b, name)
        full = torch.zeros(G * (x.numel() // b.hp.n_units), dtype=x.dtype, device=x.device)
        s["room"][name] = full
        setattr(b, name, full[:x.numel()])
    if shared:
        b.local_count = b.sel_count
    b.row_idx.zero_()
    b.val.zero_()


def prepare(case, seed):
    c = case
    if c["kind"] == "train":
        return _prepare_train(c, seed)
    h, kp, n, dim = sic.Handle(0), _kernel(c), c["n"], c["dim"]
    s = dict(case=c, h=h, kp=kp)
    if c["kind"] == "learned":
        hp = pipeline.prepare_groups(synthetic.points(n, dim, seed), kp, c["C"], c["k"])
        b = learned.LearnedFactorBuilder(h, hp, learned.Proposal(h, _params(seed), c["top"], DEV))
        b.fb = pipeline.FactorBuilder(h, b.rhp, PREC["fp32"], DEV, nnz_cap=_caps(c)[1])
        G = _caps(c)[0]
        b.buf = dict(feat=torch.zeros((G * c["C"], 8), dtype=torch.float32, device=DEV),
                     score=torch.zeros(G * c["C"], dtype=torch.float32, device=DEV),
                     out_ptr=torch.zeros(G + 1, dtype=torch.int64, device=DEV),
                     out_idx=torch.zeros(G * c["top"], dtype=torch.int32, device=DEV))
        s.update(dp=pipeline.DeviceProblem(hp, DEV), b=b, params=b.proposal.params)
        _room(s, c, ("sel_idx", "sel_count"))
    elif c["kind"] == "groups":
        hp = pipeline.prepare_groups(synthetic.points(n, dim, seed), kp, c["C"], c["k"])
        s.update(dp=pipeline.DeviceProblem(hp, DEV),
                 b=pipeline.FactorBuilder(h, hp, PREC[c["prec"]], DEV, nnz_cap=_caps(c)[1]))
        _room(s, c, ("sel_idx", "sel_count"))
    elif c["kind"] == "columns":
        hp = pipeline.prepare_columns(synthetic.points(n, dim, seed), kp, c["C"], c["k"])
        b = pipeline.FactorBuilder(h, hp, PREC[c["prec"]], DEV)
        b.row_idx.zero_()
        b.val.zero_()
        s.update(dp=pipeline.DeviceProblem(hp, DEV), b=b)
    elif c["kind"] == "partial":
        hp = pipeline.prepare_partial(synthetic.points(n, dim, seed), kp, c["C"], c["k"])
        b = pipeline.PartialFactorBuilder(h, hp, PREC[c["prec"]], DEV)
        b.nnz_cap = _caps(c)[1]
        b.row_idx, b.val = (torch.zeros(b.nnz_cap, dtype=x.dtype, device=DEV) for x in (b.row_idx, b.val))
        s.update(dp=pipeline.DeviceProblem(hp, DEV), b=b)
        _room(s, c, ("sel_idx", "sel_count", "gain"))
    elif c["kind"] == "budget":
        hp = pipeline.prepare_groups(synthetic.clustered_points(n, dim, seed), kp, c["C"], c["k"])
        s.update(dp=pipeline.DeviceProblem(hp, DEV),
                 b=pipeline.FactorBuilder(h, hp, PREC["fp32"], DEV, nnz_cap=_caps(c)[1],
                                          budget=int(c["share"] * c["k"] * n), side_fp64=True))
        _room(s, c, ("sel_idx", "sel_count", "local_count", "gain"))
    elif c["kind"] in ("refill", "apply"):
        hp = pipeline.prepare_groups(synthetic.points(n, dim, seed), kp, c["k"], c["k"])
        sel, cnt = _nearest_picks(hp)
        s["dp"] = pipeline.DeviceProblem(hp, DEV)
        if c["kind"] == "refill":
            b = pipeline.FactorBuilder(h, hp, PREC["fp64"], DEV, nnz_cap=_caps(c)[1])
            b.row_idx.zero_()
            b.val.zero_()
            b.sel_idx.copy_(torch.from_numpy(sel.reshape(-1)))
            b.sel_count.copy_(torch.from_numpy(cnt))
            s["b"] = b
        else:
            val, logv, rows, col_ptr = _factor(s["dp"].pts, c, hp.grp_ptr, sel, cnt)
            shape = (n,) if c["nrhs"] == 1 else (n, c["nrhs"])
            x = torch.from_numpy(synthetic.normal(seed, n * c["nrhs"]).reshape(shape)).to(DEV)
            s.update(col_ptr=col_ptr, row_idx=rows.to(torch.int32), val=val, x=x, y=torch.empty_like(x),
                     ws=sic._ws(sic.apply_factor_workspace(n, c["nrhs"], OPS[c["op"]]), DEV))
    elif c["kind"] == "matvec":
        shape = (n,) if c["nrhs"] == 1 else (n, c["nrhs"])
        x = torch.from_numpy(synthetic.normal(seed, n * c["nrhs"]).reshape(shape)).to(DEV)
        s.update(pts=torch.from_numpy(synthetic.points(n, dim, seed)).to(DEV), x=x, y=torch.empty_like(x))
    elif c["kind"] == "predict":
        x = synthetic.points(n + c["targets"], dim, seed)
        x_test = x[n:].copy()
        y = np.sin(7.0 * x[:n, 0]) * np.cos(5.0 * x[:n, 1]) + 0.1 * synthetic.normal(seed, n)
        s.update(x_test=x_test, model=gp.DirectedGP(h, kp, x[:n], y, c["C"], c["k"]))
    else:
        x = torch.from_numpy(synthetic.points(n + 1, dim, seed)).to(DEV)
        prec, k = PREC[c["prec"]], c["k"]
        s.update(x_train=x[:n].contiguous(), x_target=x[n].contiguous(), prec=prec,
                 idx=torch.empty(k, dtype=torch.int32, device=DEV), var=torch.zeros(k + 1, dtype=torch.float64, device=DEV),
                 count=torch.zeros(1, dtype=torch.int32, device=DEV),
                 ws=sic._ws(sic.select_single_workspace(n, k, prec), DEV))
    return s


def _prepare_train(c, seed):
    """A training batch and the optimiser's state in the middle of a run."""
    B = c["batch"]
    r = np.random.RandomState(seed % (1 << 31))
    feat = np.empty((B, 8), np.float32)
    d = np.sqrt(r.uniform(0, 1, B))
    feat[:, 2] = d
    a = r.uniform(0, 2 * np.pi, B)
    feat[:, 0], feat[:, 1] = d * np.cos(a), d * np.sin(a)
    feat[:, 3] = d + 0.3 * r.uniform(0, 1, B)
    feat[:, 4] = d * d
    feat[:, 5] = np.exp(-3 * d)
    feat[:, 6] = r.randint(8, 65, B) / 64.0
    feat[:, 7] = np.exp(-3.5 * d)
    label = (r.uniform(0, 1, B) < 0.25 * np.exp(-2 * d)).astype(np.float32)
    p = _params(seed)
    t = lambda v: torch.from_numpy(np.ascontiguousarray(v, dtype=np.float32)).to(DEV)  # noqa: E731
    n = len(p)
    return dict(case=c, h=sic.Handle(0), feat=t(feat), label=t(label), params=t(p), m=t(1e-3 * r.standard_normal(n)),
                v=t(1e-5 * (0.5 + r.uniform(0, 1, n))), grads=torch.zeros(n, dtype=torch.float32, device=DEV),
                loss=torch.zeros(1, dtype=torch.float32, device=DEV), ws=sic._ws(sic.mlp_train_workspace(B), DEV))


# -------------------------------------------------------------------- pass --

def run(state):
    s = state
    c = s["case"]
    kind = c["kind"]
    if kind in ("learned", "groups", "columns", "partial", "budget"):
        s["b"].run(s["dp"])
        b = getattr(s["b"], "fb", s["b"])
        out = dict(sel_idx=b.sel_idx, sel_count=b.sel_count, col_ptr=b.col_ptr, row_idx=b.row_idx, val=b.val,
                   logv=b.logv, sum_logv=b.sum_logv)
        out.update(s.get("room", {}))
        if kind == "learned":
            out.update(s["b"].buf)  # the network's inputs and logits, and the kept candidates
        return out
    if kind == "refill":
        b = s["b"]
        b.fill(s["dp"])
        return dict(col_ptr=b.col_ptr, row_idx=b.row_idx, val=b.val, logv=b.logv, sum_logv=b.sum_logv)
    if kind == "apply":
        sic.apply_factor(s["h"], s["col_ptr"], s["row_idx"], s["val"], OPS[c["op"]], s["x"], s["y"], s["ws"])
        return s["y"]
    if kind == "matvec":
        sic.matern_matvec(s["h"], s["pts"], s["kp"], 1e-4, PREC[c["prec"]], s["x"], s["y"])
        return s["y"]
    if kind == "predict":
        mean, var = s["model"].predict(s["x_test"])
        return dict(mean=mean, var=var, sel_idx=s["model"].last["sel_idx"], sel_count=s["model"].last["sel_count"])
    if kind == "single":
        sic.select_single(s["h"], s["x_train"], s["x_target"], s["kp"], c["k"], s["prec"], s["idx"], s["var"], s["count"], s["ws"])
        return dict(idx=s["idx"], var=s["var"], count=s["count"])
    sic.mlp_grads(s["h"], s["params"], s["feat"], s["label"], 2.0, True, s["grads"], s["loss"], s["ws"])
    sic.adamw_step(s["h"], s["params"], s["m"], s["v"], s["grads"], 100, 2e-3, wd=1e-4)
    return dict(grads=s["grads"], loss=s["loss"], params=s["params"], m=s["m"], v=s["v"])


# -------------------------------------------------------------------- work --

def work(case):
    """Bytes that have to be read or written once and arithmetic operations (2 per multiply-add; 12 per
    kernel entry)."""
    c = case
    kind = c["kind"]
    if kind == "train":
        B, P = c["batch"], 17793
        return dict(bytes=36.0 * B + 28.0 * P, flops=6.0 * B * (8 * 128 + 128 * 128 + 128))
    n, dim = c["n"], c["dim"]
    if kind == "matvec":
        return dict(bytes=8.0 * n * dim + 16.0 * n * c["nrhs"], flops=n * float(n) * (3 * dim + 12 + 2 * c["nrhs"]))
    if kind == "single":
        k = c["k"]
        return dict(bytes=8.0 * n * dim + 12.0 * k, flops=n * float(k) * (k + 16))
    if kind in ("predict", "columns"):
        u, k, C = (c["targets"] if kind == "predict" else n), c["k"], c["C"]
        sel = u * float(C) * k * (k + 16)
        fill = u * (2.0 * (k + 1) ** 3 / 6 + (k + 1) ** 2 + 6.0 * (k + 1) ** 2)
        out = u * (4.0 * k + 16) + (12.0 * u * (k + 1) if kind == "columns" else 0.0)
        return dict(bytes=8.0 * n * dim + 4.0 * u * C + out, flops=sel + fill)
    m, k = MEAN_M, c["k"]
    G = n / m
    nnz = n * (k + (m + 1) / 2)
    t = k + m
    fill = G * (t ** 3 / 3 + m * t * t + 6 * t * t)
    if kind == "apply":
        passes = 2 if c["op"] == "LLT" else 1
        return dict(bytes=12.0 * nnz + 8.0 * n + 16.0 * n * c["nrhs"], flops=2.0 * passes * nnz * c["nrhs"])
    out = 12.0 * nnz + 16.0 * n
    if kind == "refill":
        return dict(bytes=8.0 * n * dim + 4.0 * G * k + out, flops=fill)
    C = min(c["C"], c.get("top", c["C"]))
    sel = G * (2 * (C + m) * m * m / 2 + 2 * C * (k * k + k * m + 3 * k) + 12.0 * C * (k + m))
    side = G * (t ** 3 / 3 + k ** 3 / 3 + 6 * t * t) if kind == "budget" else 0.0
    net = 2.0 * G * c["C"] * (8 * 128 + 128 * 128 + 128) if kind == "learned" else 0.0
    return dict(bytes=8.0 * n * dim + 4.0 * G * (c["C"] + k) + out, flops=sel + fill + side + net)


# ------------------------------------------------------- 64-bit references --

def _matern(c, d2):
    t = math.sqrt(c["nu_x2"]) * d2.sqrt() / c["ell"]
    e = torch.exp(-t)
    if c["nu_x2"] == 1:
        return e
    return (1 + t) * e if c["nu_x2"] == 3 else (1 + t + t * t / 3) * e


def _d2(a, b):
    return (a - b).square().sum(-1)


def _factor(pts, c, grp_ptr, sel, cnt, chunk=4096):
    """The KL-optimal columns of every group: val, log v, rows (column after column: the diagonal, the other
    rows ascending) and the column pointers, from the inverse of the Cholesky factor of Theta over the
    reversed set.  sel, cnt: the picks (numpy); grp_ptr None: single columns."""
    n = pts.shape[0]
    gp_ = np.arange(n + 1) if grp_ptr is None else grp_ptr
    G, k = sel.shape
    M = int(np.max(np.diff(gp_)))
    first = torch.from_numpy(gp_[:-1]).to(pts.device)
    size = torch.from_numpy(np.diff(gp_)).to(pts.device)
    sel = torch.from_numpy(sel).to(pts.device).long()
    cnt = torch.from_numpy(np.asarray(cnt)).to(pts.device).long()
    vals, logs, rows = [], [], []
    chunk = max(1, min(chunk * 8, (1 << 27) // ((M + k) ** 2)))
    for g0 in range(0, G, chunk):
        f, z, s, q = first[g0:g0 + chunk], size[g0:g0 + chunk], sel[g0:g0 + chunk], cnt[g0:g0 + chunk]
        a = torch.arange(M, device=pts.device)[None, :]
        j = torch.arange(k, device=pts.device)[None, :]
        s = torch.where(j < q[:, None], s, torch.full_like(s, n)).sort(1).values
        ok = torch.cat([a < z[:, None], j < q[:, None]], 1)
        S = torch.where(ok, torch.cat([f[:, None] + a, s], 1), torch.zeros_like(ok, dtype=torch.long))
        X = pts[S.flip(1)]
        o = ok.flip(1)
        T = _matern(c, _d2(X[:, :, None], X[:, None])) * (o[:, :, None] & o[:, None])
        T.diagonal(dim1=1, dim2=2).copy_(1.0 + c["nugget"] * o.double())
        L = torch.linalg.cholesky(T)
        del T
        R = M + k
        e = torch.eye(R, dtype=pts.dtype, device=pts.device)[:, R - M:].expand(len(f), R, M)
        # column R-1-a of L^{-T}; flipped back: entry j >= a belongs to position S[j]
        U = torch.linalg.solve_triangular(L.transpose(1, 2), e, upper=True).flip(1).flip(2).transpose(1, 2)
        keep = ok[:, None, :] & ok[:, :M, None] & (torch.arange(R, device=pts.device)[None, :] >= a.T)[None]
        vals.append(U[keep])
        rows.append(S[:, None, :].expand(-1, M, -1)[keep])
        logs.append(2 * L.diagonal(dim1=1, dim2=2).flip(1)[:, :M][ok[:, :M]].log())
        del L, U, keep
    per = torch.repeat_interleave(size + cnt, size) - (torch.arange(n, device=pts.device) - torch.repeat_interleave(first, size))
    col_ptr = torch.zeros(n + 1, dtype=torch.int64, device=pts.device)
    col_ptr[1:] = per.cumsum(0)
    return torch.cat(vals), torch.cat(logs), torch.cat(rows), col_ptr


def _lists(ptr, idx, width, device):
    """CSR lists as a padded (units x width) array and its mask."""
    cnt = torch.from_numpy(np.diff(ptr)).to(device)
    j = torch.arange(width, device=device)[None, :]
    ok = j < cnt[:, None]
    at = (torch.from_numpy(ptr[:-1]).to(device)[:, None] + j).clamp_(max=max(len(idx) - 1, 0))
    return torch.where(ok, torch.from_numpy(idx).to(device).long()[at], torch.zeros_like(at)), ok


def _greedy(pts, c, first, size, cand, ok, k, one):
    """Greedy conditional selection of every unit in 64 bits: (picks, -1 after the last; counts).  Targets
    first .. first + size - 1; one: a single target, scored by cov^2 / var, else by var / var given the
    targets."""
    U, C = cand.shape
    M = int(size.max())
    a = torch.arange(M, device=pts.device)[None, :]
    tok = a < size[:, None]
    X, T = pts[cand], pts[torch.where(tok, first[:, None] + a, first[:, None])]
    at = torch.arange(U, device=pts.device)
    diag = 1.0 + c["nugget"]
    B = _matern(c, _d2(T[:, :, None], T[:, None])) * (tok[:, :, None] & tok[:, None])
    B.diagonal(dim1=1, dim2=2).copy_(1.0 + c["nugget"] * tok.double())
    D = _matern(c, _d2(X[:, :, None], T[:, None])) * tok[:, None]
    F2 = torch.zeros((U, C, M + k), dtype=pts.dtype, device=pts.device)
    F2[:, :, :M] = torch.linalg.solve_triangular(torch.linalg.cholesky(B), D.transpose(1, 2), upper=False).transpose(1, 2)
    F1 = torch.zeros((U, C, k), dtype=pts.dtype, device=pts.device)
    v1 = torch.full((U, C), diag, dtype=pts.dtype, device=pts.device)
    v2 = v1 - F2.square().sum(2)
    cov = D[:, :, 0].clone()
    live = ok.clone()
    picks = torch.full((U, k), -1, dtype=torch.long, device=pts.device)
    for t in range(k):
        s = cov * cov / v1 if one else v1 / v2
        q = torch.where(live, s, torch.full_like(s, -1.0)).argmax(1)
        any_ = live.any(1)
        picks[:, t] = torch.where(any_, cand[at, q], -torch.ones_like(q))
        th = _matern(c, _d2(X, X[at, q][:, None]))
        th[at, q] += c["nugget"]
        u1 = (th - (F1[:, :, :t] @ F1[at, q, :t, None])[..., 0]) / v1[at, q].sqrt()[:, None]
        if one:
            cov = cov - u1 * (cov[at, q] / v1[at, q].sqrt())[:, None]
        else:
            u2 = (th - (F2[:, :, :M + t] @ F2[at, q, :M + t, None])[..., 0]) / v2[at, q].sqrt()[:, None]
            F2[:, :, M + t] = u2
            v2 = v2 - u2 * u2
        F1[:, :, t] = u1
        v1 = v1 - u1 * u1
        live[at, q] = False
        v1 = torch.where(live, v1, torch.ones_like(v1))  # a picked row is never read again
        v2 = torch.where(live, v2, torch.ones_like(v2))
    return picks, (picks >= 0).sum(1)


def _exact_build(c, seed):
    s = prepare(c, seed)
    hp, pts = s["dp"].hp, s["dp"].pts
    k, one = hp.k, hp.grp_ptr is None
    if c["kind"] == "refill":
        picks, cnt = _nearest_picks(hp)
    else:
        cand, ok = _lists(hp.cand_ptr, hp.cand_idx, hp.max_cand, pts.device)
        gp_ = np.arange(hp.n + 1) if one else hp.grp_ptr
        first, size = torch.from_numpy(gp_[:-1]).to(pts.device), torch.from_numpy(np.diff(gp_)).to(pts.device)
        step = max(1, (1 << 28) // (hp.max_cand * (2 * k + hp.max_m)))
        got = [_greedy(pts, c, first[i:i + step], size[i:i + step], cand[i:i + step], ok[i:i + step], k, one)
               for i in range(0, hp.n_units, step)]
        picks, cnt = (torch.cat([g[i] for g in got]).cpu().numpy() for i in (0, 1))
    val, logv, _, _ = _factor(pts, c, hp.grp_ptr, picks, cnt)
    out = dict(logv=logv, sum_logv=logv.sum().reshape(1))
    # mixed-precision picks may differ from the 64-bit ones: only the sum of log v is then comparable
    if c.get("prec") == "fp32":
        return dict(sum_logv=out["sum_logv"])
    full = torch.zeros(s["b"].nnz_cap, dtype=torch.float64, device=pts.device)
    full[:val.numel()] = val
    return dict(out, val=full)


def _gelu(z):
    return 0.5 * z * (1.0 + torch.erf(z / math.sqrt(2.0)))


def _net(p):
    p = p.double()
    return (p[:1024].reshape(8, 128), p[1024:1152], p[1152:17536].reshape(128, 128), p[17536:17664], p[17664:17792], p[17792])


def _exact_learned(c, seed):
    s = prepare(c, seed)
    hp, pts = s["dp"].hp, s["dp"].pts
    W1, b1, W2, b2, w3, b3 = _net(s["params"])
    cand, ok = _lists(hp.cand_ptr, hp.cand_idx, hp.max_cand, pts.device)
    first = torch.from_numpy(hp.grp_ptr[:-1]).to(pts.device)
    size = torch.from_numpy(np.diff(hp.grp_ptr)).to(pts.device)
    feats, scores = [], []
    for i in range(0, hp.n_units, 512):
        f, z, o = first[i:i + 512], size[i:i + 512], ok[i:i + 512]
        a = torch.arange(hp.max_m, device=pts.device)[None, :]
        tok = a < z[:, None]
        X, T = pts[cand[i:i + 512]], pts[torch.where(tok, f[:, None] + a, f[:, None])]
        d = torch.empty(X.shape[:2] + (hp.max_m,), dtype=torch.float64, device=pts.device)
        for b in range(hp.max_m):
            d[:, :, b] = _d2(X, T[:, b:b + 1]).sqrt()
        d = torch.where(tok[:, None], d, torch.full_like(d, math.inf))
        near, who = d.min(2)
        C = o.sum(1)
        R = near[torch.arange(len(f), device=pts.device), (C - 1).clamp(min=0)]
        R = torch.where(R > 0, R, torch.ones_like(R))[:, None]
        at = torch.arange(len(f), device=pts.device)[:, None]
        diff = X - T[at, who]
        K = torch.where(tok[:, None], _matern(c, torch.where(tok[:, None], d, torch.zeros_like(d)).square()), torch.zeros_like(d))
        mean = (T * tok[:, :, None]).sum(1) / z[:, None]
        r = torch.arange(o.shape[1], device=pts.device, dtype=torch.float64)[None, :]
        F = torch.stack([diff[..., 0] / R, diff[..., 1] / R, near / R, _d2(X, mean[:, None]).sqrt() / R,
                         (r / C[:, None]).expand_as(near), _matern(c, near.square()), (z[:, None] / 64.0).expand_as(near),
                         K.sum(2) / z[:, None]], 2)[o]
        feats.append(F.float())
        scores.append((_gelu(_gelu(F @ W1 + b1) @ W2 + b2) @ w3 + b3).float())
    feat, score = (torch.zeros_like(s["b"].buf[name]) for name in ("feat", "score"))
    rows = int(hp.cand_ptr[-1])
    feat[:rows], score[:rows] = torch.cat(feats), torch.cat(scores)
    return dict(feat=feat, score=score)


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind in ("partial", "budget"):
        return None  # every output follows mixed-precision picks
    if kind in ("groups", "columns", "refill"):
        return _exact_build(c, seed)
    if kind == "learned":
        return _exact_learned(c, seed)
    s = prepare(c, seed)
    if kind == "apply":
        x = s["x"].reshape(c["n"], -1)
        row = s["row_idx"].long()
        col = torch.repeat_interleave(torch.arange(c["n"], device=DEV), s["col_ptr"].diff())
        if c["op"] in ("LT", "LLT"):
            x = torch.zeros_like(x).index_add_(0, col, s["val"][:, None] * x[row])
        if c["op"] in ("L", "LLT"):
            x = torch.zeros_like(x).index_add_(0, row, s["val"][:, None] * x[col])
        return x.reshape(s["x"].shape)
    if kind == "matvec":
        x, y = s["x"].reshape(c["n"], -1), []
        for i in range(0, c["n"], 1024):
            p = s["pts"][i:i + 1024]
            y.append(_matern(c, sum((p[:, None, d] - s["pts"][None, :, d]).square() for d in range(c["dim"]))) @ x)
        return (torch.cat(y) + (c["nugget"] + 1e-4) * x).reshape(s["x"].shape)
    if kind == "train":
        W = [w.clone().requires_grad_(True) for w in _net(s["params"])]
        z = _gelu(_gelu(s["feat"].double() @ W[0] + W[1]) @ W[2] + W[3]) @ W[4] + W[5]
        y = s["label"].double()
        loss = (2.0 * y * torch.nn.functional.softplus(-z) + (1 - y) * torch.nn.functional.softplus(z)).mean()
        loss.backward()
        g = torch.cat([w.grad.reshape(-1) for w in W])
        p, m, v = (s[i].double() for i in ("params", "m", "v"))
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = p - 2e-3 * (m / (1 - 0.9 ** 100) / ((v / (1 - 0.999 ** 100)).sqrt() + 1e-8) + 1e-4 * p)
        return dict(grads=g, loss=loss.detach().reshape(1), params=p, m=m, v=v)
    if kind == "single":
        if c["prec"] == "fp32":
            return None  # the picks, and with them the variances, are the mixed precision's own
        X, xt, k = s["x_train"], s["x_target"], c["k"]
        F = torch.zeros((k, c["n"]), dtype=torch.float64, device=DEV)
        var = torch.full((c["n"],), 1.0 + c["nugget"], dtype=torch.float64, device=DEV)
        cov = _matern(c, _d2(X, xt))
        out = torch.zeros(k + 1, dtype=torch.float64, device=DEV)
        out[0] = 1.0 + c["nugget"]
        live = torch.ones_like(var, dtype=torch.bool)
        for t in range(k):
            q = torch.where(live, cov * cov / var, torch.full_like(var, -1.0)).argmax()
            th = _matern(c, _d2(X, X[q]))
            th[q] += c["nugget"]
            u = (th - F[:t, q] @ F[:t]) / var[q].sqrt()
            ut = cov[q] / var[q].sqrt()
            F[t] = u
            live[q] = False
            var, cov = torch.where(live, var - u * u, torch.ones_like(var)), cov - u * ut
            out[t + 1] = out[t] - ut * ut
        return dict(var=out)
    # directed regression: the C nearest training points, the greedy picks, the posterior from them
    m = s["model"]
    xt, xr = (torch.from_numpy(v).to(DEV) for v in (s["x_test"], m.x_train))
    y = torch.from_numpy(m.y_train).to(DEV)
    pts = torch.cat([xt, xr])
    nt, C = len(xt), min(c["C"], c["n"])
    mean, var = [], []
    for i in range(0, nt, 256):
        near = torch.stack([_d2(xr, p).sort(stable=True).indices[:C] for p in xt[i:i + 256]]) + nt
        first = torch.arange(i, i + len(near), device=DEV)
        picks, _ = _greedy(pts, c, first, torch.ones_like(first), near, torch.ones_like(near, dtype=torch.bool), min(c["k"], C), True)
        P = pts[picks]
        K = _matern(c, _d2(P[:, :, None], P[:, None]))
        K.diagonal(dim1=1, dim2=2).add_(c["nugget"])
        b = _matern(c, _d2(P, xt[i:i + 256, None]))
        w = torch.linalg.solve(K, b[..., None])[..., 0]
        mean.append((w * y[picks - nt]).sum(1))
        var.append(1.0 - (w * b).sum(1))
    return dict(mean=torch.cat(mean), var=torch.cat(var))
