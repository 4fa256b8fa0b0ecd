"""Parity of pruning / compaction (sa_prune), the certificate of Prop. aoc, the duality
check (sa_certify) and the whole pipeline (sa_assign) with the oracle.

Prune decisions are compared bit for bit on the same FP64 potentials (the oracle's),
except entries whose FP64 log-domain value lies within 1e-9 of log t, where the last bit
of two different FP64 logarithms may decide.  The final assignment must have the same
exact integer product as the oracle's dense Hungarian optimum."""
import numpy as np
import pytest

import oracle
from paper_1104_3830_gb300 import api
from paper_1104_3830_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1104_3830_gb300 import build
    build.build()
    c = api.sa_create(0)
    yield c
    c.close()


def _oracle_case(n, seed, ps, dtype=np.int32, hi=1000):
    w = W.uniform(n, 1, hi, seed, dtype=dtype)
    b = oracle.log_weights(w.astype(np.int64))
    u, v, *_ = oracle.sinkhorn(b, ps, 1e-8, 20000)
    return w, b, u, v


@pytest.mark.parametrize("n,dtype,guard,t", [(256, np.int32, True, 0.0), (300, np.int16, False, 0.0),
                                             (1001, np.int16, True, 0.0), (64, np.int32, True, 0.5),
                                             (5, np.int16, True, 0.0)])
def test_prune_matches_oracle(ctx, n, dtype, guard, t):
    ps = [1.0, 2.0, 4.0, 8.0, 16.0]
    w, b, u, v = _oracle_case(n, 300 + n, ps, dtype)
    d = api.to_device(w)
    rp, col, wv, ub = api.sa_prune(ctx, d, ps[-1], torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda(), t, guard)
    mask_g = np.zeros((n, n), dtype=bool)
    rows = np.repeat(np.arange(n), np.diff(rp))
    mask_g[rows, col] = True
    assert np.all(np.diff(col[rp[:-1].clip(max=len(col) - 1)]) >= -n)  # well formed
    for i in range(n):
        assert np.all(np.diff(col[rp[i]:rp[i + 1]]) > 0)
    assert np.array_equal(wv, w[rows, col])
    tt = t if t > 0 else 1.0 / n
    mask_o = oracle.prune_mask(b, ps[-1], u, v, tt, guard)
    e = ps[-1] * b - u[:, None] - v[None, :]
    near = np.abs(e - np.log(tt)) < 1e-9
    assert np.array_equal(mask_g & ~near, mask_o & ~near)
    if guard:
        assert mask_g.any(axis=1).all() and mask_g.any(axis=0).all()
    assert abs(ub - oracle.log_ub(b, ps[-1], v)) < 1e-9 * max(1.0, abs(ub))


def test_certify_counts_like_oracle(ctx):
    w = W.uniform(200, 1, 1000, 500, dtype=np.int16)
    b = oracle.log_weights(w.astype(np.int64))
    perm, al, be, _ = oracle.hungarian(b)
    d = api.to_device(w)
    nv, _ = api.sa_certify(ctx, d, al, be, 1e-9)
    assert nv == 0
    bb = b.copy()
    bb[np.arange(200), perm] = -np.inf
    _, al2, be2, _ = oracle.hungarian(bb)
    nv2, (rp, col, wv) = api.sa_certify(ctx, d, al2, be2, 1e-9)
    cnt, _ = oracle.dual_violations(b, al2, be2, 1e-9)
    assert nv2 == cnt and rp[-1] == cnt
    rows = np.repeat(np.arange(200), np.diff(rp))
    assert np.all(b[rows, col] - al2[rows] - be2[col] > 1e-9)
    assert np.array_equal(wv, w[rows, col])


@pytest.mark.parametrize("case", ["c1", "uniform777", "planted2048", "tied1024", "zipf300"])
def test_assign_is_exactly_optimal(ctx, case):
    if case == "c1":
        w, ps = W.c1()
    elif case == "uniform777":
        w, ps = W.uniform(777, 1, 1000, 600, dtype=np.int16), [2.0 ** k for k in range(8)]
    elif case == "planted2048":
        w, pi, _ = W.planted(2048, 601)
        ps = [2.0 ** k for k in range(10)]
    elif case == "tied1024":
        w, pi, _ = W.planted(1024, 602, tied_frac=0.01)
        ps = [2.0 ** k for k in range(10)]
    else:
        w, ps = W.zipf(300, 1.2, 30000, 603), [2.0 ** k for k in range(9)]
    d = api.to_device(w)
    r = api.sa_assign(ctx, d, ps, 1e-6, 2000)
    perm = r["perm"]
    assert sorted(perm) == list(range(len(perm)))
    b = oracle.log_weights(w.astype(np.int64))
    if case.startswith("planted") or case.startswith("tied"):
        ref = oracle.perm_weight_exact(w, pi)
    else:
        ref = oracle.perm_weight_exact(w, oracle.hungarian(b)[0])
    assert oracle.perm_weight_exact(w, perm) == ref
    assert r["gamma"] >= 1 - 1e-9
    assert r["nnz_first"] < w.size


def test_assign_host_equals_device(ctx):
    w, ps = W.c1()
    d = api.to_device(w)
    r1 = api.sa_assign(ctx, d, ps)
    r2 = api.sa_assign_host(ctx, w, ps)
    assert oracle.perm_weight_exact(w, r1["perm"]) == oracle.perm_weight_exact(w, r2["perm"])
    assert r1["scale"]["sweeps_total"] == r2["scale"]["sweeps_total"]


def test_narrowing(ctx):
    w = W.uniform(100, 1, 32767, 700, dtype=np.int32)
    src = torch.from_numpy(w).cuda()
    dst = torch.zeros((100, 104), dtype=torch.int16, device="cuda")[:, :100]
    assert api.sa_narrow_i32_to_i16(ctx, src, dst) == 0
    assert np.array_equal(dst.cpu().numpy().astype(np.int32), w)
    src[3, 4] = 40000
    assert api.sa_narrow_i32_to_i16(ctx, src, dst) == 1


@pytest.mark.parametrize("n,dtype,hi,padded,zeros", [(1, np.int16, 9, True, False), (7, np.int32, 50, False, True),
                                                     (255, np.int16, 1000, True, True), (256, np.int32, 1000, True, False),
                                                     (257, np.int16, 1000, False, True), (1030, np.int32, 2 ** 30, True, True),
                                                     (1100, np.int16, 4, True, True)])
@pytest.mark.parametrize("guard", [True, False])
def test_prune_and_certify_edges(ctx, n, dtype, hi, padded, zeros, guard):
    """Edges of the scans' tiles (256 columns, 32 x 32 keep bits, up to 256 rows a block), rows
    off 16-byte boundaries, absent entries and many equal weights (the guards' lowest index)."""
    rng = np.random.default_rng(n)
    w = rng.integers(1, hi + 1, (n, n)).astype(dtype)
    if zeros:
        w[rng.random((n, n)) < 0.3] = 0
        w[np.arange(n), np.arange(n)] = 1
    p = 4.0
    b = oracle.log_weights(w.astype(np.int64))
    # potentials with all but three bits of their mantissa zero, so that equal weights of equal
    # columns tie exactly in FP32 as in FP64
    u = np.round(p * np.log(max(hi, 2)) * 4) / 4 + rng.integers(-3, 4, n) * 0.25
    v = rng.integers(-2, 3, n) * 0.25
    d = api.to_device(w) if padded else torch.from_numpy(w).cuda()
    rp, col, wv, ub = api.sa_prune(ctx, d, p, torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda(), 0.0, guard)
    rows = np.repeat(np.arange(n), np.diff(rp))
    assert rp[0] == 0 and rp[-1] == len(col) and np.array_equal(wv, w[rows, col])
    for i in range(n):
        assert np.all(np.diff(col[rp[i]:rp[i + 1]]) > 0)
    got = np.zeros((n, n), dtype=bool)
    got[rows, col] = True
    e = p * b - u[:, None] - v[None, :]
    above = e >= np.log(1.0 / n)
    near = np.abs(e - np.log(1.0 / n)) < 1e-9
    assert np.array_equal((got & above) & ~near, above & ~near)
    extra = got & ~above & ~near
    if guard:   # beyond the threshold only row and column maxima, one a row and column
        m = (e >= e.max(1, keepdims=True) - 2e-4) | (e >= e.max(0, keepdims=True) - 2e-4)
        assert not np.any(extra & ~m) and extra.sum() <= 2 * n
        assert got.any(1).all() and got.any(0).all()
    else:
        assert not extra.any()
    assert abs(ub - oracle.log_ub(b, p, v)) < 1e-9 * max(1.0, abs(ub)) + 1e-4 * n / p
    # duals on the row maxima but for a few rows
    beta = v / p
    alpha = (b - beta).max(1)
    alpha[::3] -= 0.37
    nv, (arp, acol, aw) = api.sa_certify(ctx, d, alpha, beta, 1e-9, max_add=n * n)
    viol = b - alpha[:, None] - beta > 1e-9
    assert nv == viol.sum() == arp[-1]
    got = np.zeros((n, n), dtype=bool)
    ar = np.repeat(np.arange(n), np.diff(arp))
    got[ar, acol] = True
    assert np.array_equal(got, viol) and np.array_equal(aw, w[ar, acol])
