"""The calls whose speed matters to a user of this library, one case each.

listed()            the cases; draw(rng) gives further ones of the same ranges
prepare(case, seed) the inputs, and the context a program keeps, on the GPU
run(state)          one call through the public entry points, and its outputs
exact(case, seed)   the same outputs in 64 bits from plain torch, where they have one
work(case)          bytes and operations one call cannot do without

Weights are drawn on the GPU from the distributions of ``workloads.py`` (uniform, planted
permutation, Zipf, Euclidean points).

The scaling cases run a fixed budget of sweeps at every p (a tolerance below what FP32
sums resolve), the way a preprocessing step with a time budget runs, so that two builds
compare the same iterate.  Potentials are defined up to a constant, (u + c, v - c), so they
come back in one gauge, sum_j v_j = 0, as one vector (u, v).  The whole calls (assignment,
Algorithm 1) stop on their tolerance and return what a user keeps: the permutation, its
weight and the certificate.  Lists of a length that the values decide go into buffers of
the program's own.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_1104_3830_gb300 import _lib as L
from paper_1104_3830_gb300 import api

FIXED_BUDGET_TOL = 1e-12
DEV = "cuda:0"
_CSR_CAP = 1024   # entries a row of a reduced instance that a program makes room for


def listed():
    return [
        # the smallest single matrix: every sweep is latency (grid barriers, one row pass)
        dict(name="scale 256 int32", kind="scale", n=256, dist="uniform", hi=1000, bits=32, top=8, sweeps=50),
        # a large serving request: Zipf weights, a matrix of 4 MB of K
        dict(name="scale 1000 int16 zipf", kind="scale", n=1000, dist="zipf", hi=30000, bits=16, top=8, sweeps=50),
        # the middle of the range at a ragged width: distances between points, 32-bit weights
        dict(name="scale 2047 int32 euclid", kind="scale", n=2047, dist="euclid", hi=1 << 20, bits=32, top=8, sweeps=40),
        # the headline matrix: planted permutation, K twice the L2
        dict(name="scale 8192 int16 planted", kind="scale", n=8192, dist="planted", hi=10000, bits=16, top=9, sweeps=20),
        # the largest single matrix (the precision workload's): 1.6 GB of K
        dict(name="scale 20000 int16", kind="scale", n=20000, dist="uniform", hi=32767, bits=16, top=8, sweeps=8),
        # thousands of small independent instances in one call
        dict(name="batch 4096 int32", kind="batch", k=4096, lo=16, n=512, hi=1000, bits=32, top=7, sweeps=32),
        # the row and column sums of a scaling in 64 bits, as a user checks a result
        dict(name="verify 8192 int16", kind="verify", n=8192, dist="planted", hi=10000, bits=16, p=128.0),
        # the reduced instance of a scaled matrix, to the host as CSR
        dict(name="prune 8192 int16", kind="prune", n=8192, dist="uniform", hi=32767, bits=16, p=512.0),
        # the optimality check of host duals against a whole matrix of ragged width
        dict(name="certify 5001 int32", kind="certify", n=5001, dist="uniform", hi=1000000, bits=32, p=64.0),
        # a matrix in host memory to its certified optimal permutation, the end-to-end call
        dict(name="assign host 4096 int16", kind="assign", n=4096, dist="planted", hi=10000, bits=16, top=7, sweeps=500,
             kernel="auto", host=True),
        # the same with the Newton scaling on a device matrix
        dict(name="assign newton 3001 int32", kind="assign", n=3001, dist="planted", hi=10000, bits=32, top=9, sweeps=500,
             kernel="newton", host=False),
        # the paper's own experiment: Algorithm 1 with adaptive p on the Euclidean matrix
        dict(name="algorithm1 1000 euclid", kind="alg1", n=1000, dist="euclid", hi=1 << 20, bits=32, kernel="auto"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["scale", "scale", "scale", "batch", "verify", "prune", "certify", "assign", "alg1"])
    if kind == "batch":
        c = dict(kind=kind, k=_log_int(rng, 16, 4096), lo=rng.choice([16, 24, 32]), n=_log_int(rng, 64, 512),
                 hi=rng.choice([1000, 30000]), bits=rng.choice([16, 32]), top=rng.choice([6, 7]),
                 sweeps=rng.randint(8, 32))
        return c
    dist = rng.choice(["uniform", "zipf", "planted", "euclid"])
    if kind in ("assign", "prune", "certify") and dist == "zipf":
        dist = "uniform"   # equal weights everywhere: many optima, rows that are kept whole
    bits = 32 if dist == "euclid" else rng.choice([16, 32])
    hi = {"uniform": 32767 if bits == 16 else 1000000, "zipf": 30000, "planted": 10000, "euclid": 1 << 20}[dist]
    if kind == "scale":
        n, top = _log_int(rng, 64, 20000), rng.choice([7, 8, 9])
        most = 9 * 8 * 20000 ** 2 // ((top + 1) * n * n)
        return dict(kind=kind, n=n, dist=dist, hi=hi, bits=bits, top=top, sweeps=max(2, min(rng.randint(8, 48), most)))
    if kind == "assign":
        kernel = rng.choice(["auto", "newton"])
        return dict(kind=kind, n=_log_int(rng, 256, 4096), dist="planted", hi=10000, bits=rng.choice([16, 32]),
                    top=rng.choice([6, 7]), sweeps=500, kernel=kernel, host=rng.choice([True, False]))
    if kind == "alg1":
        return dict(kind=kind, n=_log_int(rng, 200, 1500), dist="euclid", hi=1 << 20, bits=32, kernel="auto")
    return dict(kind=kind, n=_log_int(rng, 200, 8192), dist=dist, hi=hi, bits=bits, p=float(2 ** rng.randint(6, 9)))


# ---- inputs ------------------------------------------------------------------------------

def _rows(n):
    return max(1, (1 << 25) // n)


def _weights(case, seed):
    """The n x n weights on the GPU, rows padded to 16 bytes, and the planted permutation."""
    n, dtype = case["n"], torch.int16 if case["bits"] == 16 else torch.int32
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    per = 128 // case["bits"]
    buf = torch.zeros((n, -(-n // per) * per), dtype=dtype, device=DEV)
    w = buf[:, :n]
    pi = None
    if case["dist"] == "euclid":
        x, y = (torch.rand((n, 3), generator=g, device=DEV, dtype=torch.float64) for _ in range(2))
        for r in range(0, n, _rows(n)):
            d = (x[r:r + _rows(n), None, :] - y[None, :, :]).square().sum(2).sqrt()
            w[r:r + _rows(n)] = torch.round(case["hi"] * torch.exp(-d)).clamp(min=1).to(dtype)
    elif case["dist"] == "zipf":
        k = torch.arange(1, case["hi"] + 1, device=DEV, dtype=torch.float64)
        cdf = torch.cumsum(k ** -1.2, 0)
        cdf /= cdf[-1].clone()
        for r in range(0, n, _rows(n)):
            u = torch.rand((min(_rows(n), n - r), n), generator=g, device=DEV, dtype=torch.float64)
            w[r:r + _rows(n)] = (torch.searchsorted(cdf, u, right=True).clamp(max=case["hi"] - 1) + 1).to(dtype)
    else:
        top = 9500 if case["dist"] == "planted" else case["hi"]
        for r in range(0, n, _rows(n)):
            w[r:r + _rows(n)] = torch.randint(1, top + 1, (min(_rows(n), n - r), n), generator=g, device=DEV,
                                              dtype=torch.int32).to(dtype)
        if case["dist"] == "planted":   # each row's largest weight + 500 on a hidden permutation
            pi = torch.randperm(n, generator=g, device=DEV)
            rows = torch.arange(n, device=DEV)
            w[rows, pi] = 0
            w[rows, pi] = (w.amax(1).to(torch.int32) + 500).to(dtype)
    return w, pi


def _schedule(case):
    return [2.0 ** k for k in range(case["top"] + 1)]


def _sinkhorn64(w, ps, sweeps):
    """The sweeps of the log-domain iteration in 64 bits: (u, v) after `sweeps` at each p."""
    n = w.size(0)
    b = torch.log(w.to(torch.float64))
    v = torch.zeros(n, dtype=torch.float64, device=w.device)
    for k, p in enumerate(ps):
        if k:
            v = v * (p / ps[k - 1])
        K = b * p
        K -= v
        m = K.amax(1)
        K -= m[:, None]
        K.exp_()
        c = torch.ones_like(v)
        for _ in range(sweeps):
            s = K @ c
            c = 1.0 / (K.T @ (1.0 / s))
        u = m + torch.log(s)
        v = v - torch.log(c)
    return u, v


def _potentials(w, p):
    """Potentials of X(p) as a scaling that stops early leaves them, with FP32 accuracy."""
    ps = [2.0 ** k for k in range(int(math.log2(p)) + 1)]
    return tuple(x.float().double() for x in _sinkhorn64(w, ps, 6))


def _duals(case, seed):
    """Host duals near the optimum: v/p, and row maxima of log w - beta but for one row in
    fifty, whose third largest leaves two violations of the certificate."""
    w, _ = _weights(case, seed)
    _, v = _potentials(w, case["p"])
    beta = v / case["p"]
    red = torch.log(w.to(torch.float64)) - beta
    top3 = torch.topk(red, 3, dim=1).values
    alpha = top3[:, 0].clone()
    alpha[::50] = top3[::50, 2]
    return w, alpha, beta


def _sizes(case):
    rng = np.random.default_rng(case["k"])
    lo, hi = case["lo"], case["n"]
    return np.clip(np.exp(rng.uniform(math.log(lo), math.log(hi + 1), case["k"])).astype(np.int64), lo, hi)


def _pack(case, seed):
    """k instances of log-uniform size, one after the other in a buffer, rows of 16 bytes."""
    ns = _sizes(case)
    per = 128 // case["bits"]
    lds = (ns + per - 1) // per * per
    offs = np.concatenate([[0], np.cumsum(lds * ns)])
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    flat = torch.randint(1, case["hi"] + 1, (int(offs[-1]),), generator=g, device=DEV, dtype=torch.int32)
    return ns, lds, offs[:-1], flat.to(torch.int16 if case["bits"] == 16 else torch.int32)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, kind=kind, ctx=api.sa_create(0))
    if kind == "batch":
        ns, lds, offs, flat = _pack(case, seed)
        s["w"] = flat
        s["ptrs"] = torch.from_numpy(flat.data_ptr() + offs * flat.element_size()).to(DEV)
        s["n"] = torch.from_numpy(ns.astype(np.int32)).to(DEV)
        s["ld"] = torch.from_numpy(lds).to(DEV)
        s["off"] = torch.from_numpy(np.concatenate([[0], np.cumsum(ns)[:-1]])).to(DEV)
        s["member"] = torch.from_numpy(np.repeat(np.arange(len(ns)), ns)).to(DEV)
        s["count"] = torch.from_numpy(ns.astype(np.float64)).to(DEV)
        s["uv"] = torch.zeros(2 * int(ns.sum()), dtype=torch.float64, device=DEV)
        s["u"], s["v"] = s["uv"].chunk(2)
        s["opts"] = L.make_opts(_schedule(case), FIXED_BUDGET_TOL, case["sweeps"])
        return s
    if kind == "certify":
        s["w"], alpha, beta = _duals(case, seed)
        s["alpha"], s["beta"] = alpha.cpu().numpy(), beta.cpu().numpy()
        s["col"], s["weight"] = (np.zeros(1 << 16, dtype=np.int32) for _ in range(2))
        return s
    s["w"], _ = _weights(case, seed)
    if kind == "scale":
        s["uv"] = torch.zeros(2 * case["n"], dtype=torch.float64, device=DEV)
        s["u"], s["v"] = s["uv"].chunk(2)
    if kind == "prune":
        s["col"], s["weight"] = (np.zeros(min(_CSR_CAP, case["n"]) * case["n"], dtype=np.int32) for _ in range(2))
    if kind in ("verify", "prune"):
        s["u"], s["v"] = _potentials(s["w"], case["p"])
    if case.get("host"):
        pinned = torch.empty(s["w"].shape, dtype=s["w"].dtype, pin_memory=True)
        pinned.copy_(s["w"])
        s["w"] = pinned
        s["host"] = pinned.numpy()
    return s


def run(s):
    case, kind, ctx = s["case"], s["kind"], s["ctx"]
    if kind == "scale":
        u, v, _ = api.sa_scale(ctx, s["w"], _schedule(case), FIXED_BUDGET_TOL, case["sweeps"], u=s["u"], v=s["v"])
        mean = v.mean()
        u += mean
        v -= mean
        return s["uv"]
    if kind == "batch":
        ptr = {x: ctypes.c_void_p(s[x].data_ptr()) for x in ("ptrs", "n", "ld", "off", "u", "v")}
        rc = L.lib().sa_batch_scale(ctx.handle, case["k"], ptr["ptrs"], ptr["n"], ptr["ld"], ptr["off"],
                                    L.SA_I16 if case["bits"] == 16 else L.SA_I32, ctypes.byref(s["opts"]), ptr["u"],
                                    ptr["v"], None, None)
        if rc != L.SA_E_NOT_CONVERGED:   # a fixed budget ends on its cap
            L.check(rc)
        mean = torch.zeros_like(s["count"]).index_add_(0, s["member"], s["v"]).div_(s["count"])[s["member"]]
        s["u"] += mean
        s["v"] -= mean
        return s["uv"]
    if kind == "verify":
        row_err, col_err, rows, cols = api.sa_verify(ctx, s["w"], case["p"], s["u"], s["v"], want_sums=True)
        return row_err, col_err, rows, cols
    if kind == "prune":
        row_ptr, col, weight, log_ub = api.sa_prune(ctx, s["w"], case["p"], s["u"], s["v"])
        s["col"][:len(col)] = col
        s["weight"][:len(col)] = weight
        return row_ptr, s["col"], s["weight"], log_ub
    if kind == "certify":
        count, (row_ptr, col, weight) = api.sa_certify(ctx, s["w"], s["alpha"], s["beta"])
        s["col"][:len(col)] = col
        s["weight"][:len(col)] = weight
        return count, row_ptr, s["col"], s["weight"]
    if kind == "assign":
        if case["host"]:
            r = api.sa_assign_host(ctx, s["host"], _schedule(case), 1e-6, case["sweeps"], kernel=case["kernel"])
        else:
            r = api.sa_assign(ctx, s["w"], _schedule(case), 1e-6, case["sweeps"], kernel=case["kernel"])
        return r["perm"], r["sum_log_w"], r["log_ub"]
    r = api.sa_algorithm1(ctx, s["w"], opt_ratio=2.0, p0=100.0, dp=50.0, max_rounds=30, kernel=case["kernel"])
    return r["perm"], r["sum_log_w"], r["gamma"], r["p_final"], r["rounds"]


# ---- what the outputs are in 64 bits -----------------------------------------------------

def _batch64(case, seed):
    """Fixed-budget scaling of every instance: instances of like size padded and run together."""
    ns, lds, offs, flat = _pack(case, seed)
    starts = np.concatenate([[0], np.cumsum(ns)[:-1]])
    U = torch.zeros(int(ns.sum()), dtype=torch.float64, device=DEV)
    V = torch.zeros_like(U)
    ps = _schedule(case)
    order = np.argsort(ns, kind="stable")
    for at in range(0, len(order), 128):
        some = order[at:at + 128]
        m = int(ns[some].max())
        b = torch.full((len(some), m, m), -math.inf, dtype=torch.float64, device=DEV)
        real = torch.zeros((len(some), m), dtype=torch.bool, device=DEV)
        for q, i in enumerate(some):
            n, ld, o = int(ns[i]), int(lds[i]), int(offs[i])
            b[q, :n, :n] = torch.log(flat[o:o + n * ld].view(n, ld)[:, :n].to(torch.float64))
            real[q, :n] = True
        one = torch.ones((), dtype=torch.float64, device=DEV)
        v = torch.zeros((len(some), m), dtype=torch.float64, device=DEV)
        for k, p in enumerate(ps):
            if k:
                v = v * (p / ps[k - 1])
            e = b * p - v[:, None, :]
            mx = torch.where(real, e.amax(2), 0.0 * one)
            K = torch.exp(e - mx[:, :, None])
            c = real.to(torch.float64)
            for _ in range(case["sweeps"]):
                s = torch.where(real, torch.bmm(K, c[:, :, None])[:, :, 0], one)
                t = torch.bmm((real / s)[:, None, :], K)[:, 0, :]
                c = torch.where(real, 1.0 / torch.where(real, t, one), 0.0 * one)
            u = mx + torch.log(s)
            v = torch.where(real, v - torch.log(torch.where(real, c, one)), 0.0 * one)
        for q, i in enumerate(some):
            n, o = int(ns[i]), int(starts[i])
            mean = v[q, :n].mean()
            U[o:o + n] = u[q, :n] + mean
            V[o:o + n] = v[q, :n] - mean
    return torch.cat([U, V])


def exact(case, seed):
    kind = case["kind"]
    if kind == "scale":
        w, _ = _weights(case, seed)
        u, v = _sinkhorn64(w, _schedule(case), case["sweeps"])
        return torch.cat([u + v.mean(), v - v.mean()])
    if kind == "batch":
        return _batch64(case, seed)
    if kind == "verify":
        w, _ = _weights(case, seed)
        u, v = _potentials(w, case["p"])
        x = torch.exp(case["p"] * torch.log(w.to(torch.float64)) - u[:, None] - v)
        rows, cols = x.sum(1), x.sum(0)
        return float((rows - 1).abs().max()), float((cols - 1).abs().max()), rows, cols
    if kind == "prune":
        w, _ = _weights(case, seed)
        u, v = _potentials(w, case["p"])
        e = case["p"] * torch.log(w.to(torch.float64)) - v
        return None, None, None, float((e.amax(1).sum() + v.sum()) / case["p"])
    if kind == "assign":
        w, pi = _weights(case, seed)
        return None, float(torch.log(w.gather(1, pi[:, None]).to(torch.float64)).sum()), None
    return None


# ---- the work of one call ----------------------------------------------------------------

def work(case):
    kind, sz = case["kind"], case["bits"] // 8
    if kind == "batch":
        ns = _sizes(case).astype(np.float64)
        entries, vecs = float((ns * ns).sum()), float(ns.sum())
    else:
        entries, vecs = float(case["n"]) ** 2, float(case["n"])
    if kind in ("scale", "batch"):
        # per p one evaluation of the entries (multiply, add), per sweep two multiply-adds
        return dict(bytes=entries * sz + 16 * vecs, flops=(case["top"] + 1) * (4.0 * case["sweeps"] + 2) * entries)
    if kind == "verify":
        return dict(bytes=entries * sz + 32 * vecs, flops=6 * entries)
    if kind == "prune":
        return dict(bytes=entries * sz + 24 * vecs, flops=4 * entries)
    if kind == "certify":
        return dict(bytes=entries * sz + 24 * vecs, flops=2 * entries)
    # the calls that stop on a tolerance: at least one sweep at each p, one prune, one check
    steps = case["top"] + 1 if kind == "assign" else 1
    return dict(bytes=entries * sz + 4 * vecs, flops=(6.0 * steps + 6) * entries)
