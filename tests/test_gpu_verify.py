"""sa_verify's sums in fixed point against the definition in extended precision.

Tolerance, derived: each term 2^E carries at most the error of E times ln 2.  E's parts are
rounded at 2^-53 of their magnitude M (p log2 w, |U|, |V|) or at 2^-57, a handful of times,
and the sums add at most n roundings of 2^-53.  8 (M + 16) 2^-53 + n 2^-53 relative to the sum
of the terms covers both the fixed-point form and the FP64 formula it stands in for."""
import numpy as np
import pytest

from paper_1104_3830_gb300 import api

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


def _case(n, dtype, hi, p, seed, scale=1.0):
    rng = np.random.default_rng(seed)
    w = rng.integers(0, hi + 1, (n, n)).astype(dtype)
    w[rng.integers(0, n, n), rng.integers(0, n, n)] = hi      # the largest weight is there
    # row maxima of p log w near u, some rows and columns far off: sums from tiny to huge
    u = p * np.log(hi) + rng.normal(0.0, 3.0, n) * scale
    v = rng.normal(0.0, 2.0, n) * scale
    return w, u, v


def _exact(w, p, u, v):
    L = np.longdouble
    with np.errstate(divide="ignore"):
        e = L(p) * np.log(w.astype(L)) - u.astype(L)[:, None] - v.astype(L)
    x = np.exp(e)
    return x.sum(1), x.sum(0)


@pytest.mark.parametrize("n,dtype,hi,p,scale,padded", [
    (1, np.int32, 77, 8.0, 1.0, False),            # one entry
    (7, np.int16, 32767, 64.0, 1.0, True),         # less than one tile of columns
    (33, np.int32, 1 << 20, 16.0, 1.0, False),     # one row past a warp's lanes
    (159, np.int16, 32767, 8.0, 1.0, True),
    (160, np.int16, 32767, 1.0, 1.0, True),
    (257, np.int16, 30000, 64.0, 1.0, True),       # a tile and one column
    (513, np.int32, 1000, 256.0, 1.0, True),
    (255, np.int32, 2 ** 31 - 1, 3.7, 1.0, True),  # the largest weights, p with a full mantissa
    (700, np.int32, 1 << 20, 512.0, 1.0, True),    # weights above the table
    (333, np.int16, 999, 128.0, 100.0, True),      # sums over most of the exponent range
    (301, np.int16, 1000, 16.0, 1.0, False),       # rows off 16-byte boundaries
    (300, np.int32, 32768, 1e5, 1.0, True),        # too large for the fixed point
])
def test_verify_against_extended_precision(ctx, n, dtype, hi, p, scale, padded):
    w, u, v = _case(n, dtype, hi, p, 900 + n, scale)
    d = api.to_device(w) if padded else torch.from_numpy(w).cuda()
    er, ec, rows, cols = api.sa_verify(ctx, d, p, torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda(), want_sums=True)
    rows, cols = rows.cpu().numpy(), cols.cpu().numpy()
    r, c = _exact(w, p, u, v)
    m = max(p * np.log2(hi), np.abs(u).max() * 1.5, np.abs(v).max() * 1.5)
    tol = (8 * (m + 16) + n) * 2.0 ** -53
    for got, want in ((rows, r), (cols, c)):
        over = want > np.finfo(np.float64).max        # such a sum is inf in FP64
        assert np.all(np.isinf(got[over]))
        got, want = got[~over], want[~over]
        assert np.max(np.abs(got - want) / (want + 1e-300)) < tol
    assert er == np.max(np.abs(rows - 1)) and ec == np.max(np.abs(cols - 1))


def test_verify_potentials_that_are_not_finite(ctx):
    w, u, v = _case(200, np.int16, 1000, 4.0, 77)
    u[3] = np.inf                      # x = 0 along the row
    d = api.to_device(w)
    _, _, rows, cols = api.sa_verify(ctx, d, 4.0, torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda(), want_sums=True)
    r, c = _exact(w, 4.0, u, v)
    assert float(rows[3]) == 0.0
    assert np.allclose(rows.cpu().numpy(), r.astype(float), rtol=1e-12)
    assert np.allclose(cols.cpu().numpy(), c.astype(float), rtol=1e-12)


@pytest.mark.parametrize("p", [3.0, 512.0])
def test_verify_weights_above_the_table(ctx, p):
    """One entry a row and column, so that a sum is one term 2^E of a weight of 2^15 .. 2^31 - 1.  E is a
    sum of numbers rounded to units of 2^-F (the table's, the series', U and V in two parts each: at
    most 3 units), F as the kernel chooses it; 2^E adds a few roundings of 2^-53."""
    n = 2000
    rng = np.random.default_rng(12)
    wv = np.floor(2.0 ** rng.uniform(15.0, 31.0, n)).astype(np.int64)
    wv[:6] = [32768, 32769, 65535, 65536, 2 ** 31 - 1, 2 ** 30]
    w = np.zeros((n, n), dtype=np.int32)
    pi = rng.permutation(n)
    w[np.arange(n), pi] = wv
    v = rng.normal(0.0, 2.0, n)
    u = p * np.log(wv) - v[pi] + rng.normal(0.0, 1.0, n)
    _, _, rows, cols = api.sa_verify(ctx, api.to_device(w), p, torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda(),
                                     want_sums=True)
    L = np.longdouble
    x = np.exp(L(p) * np.log(wv.astype(L)) - u.astype(L) - v[pi].astype(L))
    m = max(p * 31, np.abs(u).max() * 1.4427, np.abs(v).max() * 1.4427)
    tol = 3 * 2.0 ** -(60 - int(np.floor(np.log2(m + 1)))) * np.log(2) + 6 * 2.0 ** -53
    assert np.max(np.abs(rows.cpu().numpy() - x) / x) < tol
    assert np.max(np.abs(cols.cpu().numpy()[pi] - x) / x) < tol
