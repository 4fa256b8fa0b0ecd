"""The step kernel on a K that stays on the chip (matrices up to n of about 3300) at the edges of
its shapes.  Tolerances are the step path's (test_gpu_step): both sides stop within
tol = 1e-6 of bistochastic, so X agrees with the oracle's to 8e-6 max(x, 1/n) and its FP64 sums
are within tol + 1e-6 of one."""
import numpy as np
import pytest

import oracle
from paper_1104_3830_gb300 import _lib as L
from paper_1104_3830_gb300 import api
from paper_1104_3830_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SUM_BOUND = 2e-6


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1104_3830_gb300 import build
    build.build()
    c = api.sa_create(0)
    yield c
    c.close()


def _check(ctx, w, d, ps, u, v, info, against_oracle):
    assert info["status"] == 0 and info["kernel_used"] == 3, info
    assert max(api.sa_verify(ctx, d, ps[-1], u, v)) < SUM_BOUND
    if against_oracle:
        b = oracle.log_weights(w.astype(np.int64))
        uo, vo, _, _, st = oracle.sinkhorn(b, ps, 1e-6, 20000)
        assert st == 0
        x, xo = (oracle.xmatrix(b, ps[-1], *uv) for uv in ((u.cpu().numpy(), v.cpu().numpy()), (uo, vo)))
        assert np.all(np.abs(x - xo) <= 8e-6 * np.maximum(xo, 1.0 / w.shape[0]) + 1e-9)


# one row, one block and several, the edges of the widths (512, 1024, 2048 columns of threads),
# of the rows in registers (8 a block up to n = 1216, 14 up to 2048) and near the largest that fit
@pytest.mark.parametrize("n", [1, 5, 16, 71, 511, 513, 1001, 1216, 1217, 2047, 2050, 3333])
@pytest.mark.parametrize("dtype", [np.int16, np.int32])
def test_resident_shapes(ctx, n, dtype):
    w = W.uniform(n, 1, 30000 if dtype == np.int16 else 1 << 20, 40 + n, dtype=dtype)
    if n > 16:   # absent entries and columns of very different mass
        w[:: 3, 1:: 7] = 0
        w[:, n // 2:] = np.maximum(w[:, n // 2:] >> 6, (w[:, n // 2:] > 0).astype(dtype))
    d = api.to_device(w)
    ps = [1.0, 2.0, 4.0, 8.0]
    u, v, info = api.sa_scale(ctx, d, ps, 1e-6, 20000, kernel="step")
    _check(ctx, w, d, ps, u, v, info, n <= 1217)


@pytest.mark.parametrize("grid", [1, 8, 20, 76])
def test_resident_capped_grids(ctx, grid):
    """Longer stripes on fewer blocks (and the streaming kernel where they do not fit)."""
    n = 300
    w = W.uniform(n, 1, 1000, 43, dtype=np.int16)
    d = api.to_device(w)
    ps = [1.0, 4.0]
    api.sa_set_option(ctx, "max_grid", grid)
    try:
        u, v, info = api.sa_scale(ctx, d, ps, 1e-6, 20000, kernel="step")
    finally:
        api.sa_set_option(ctx, "max_grid", 0)
    _check(ctx, w, d, ps, u, v, info, True)


def test_resident_resume_keep_and_large_steps(ctx):
    n = 700
    w = W.uniform(n, 1, 1000, 41, dtype=np.int16)
    d = api.to_device(w)
    ps = [1.0, 2.0, 4.0, 8.0, 16.0]
    u, v, _ = api.sa_scale(ctx, d, ps[:3], 1e-6, 20000, kernel="step")
    u, v, info = api.sa_scale(ctx, d, ps, 1e-6, 20000, kernel="step", resume_from=3, u=u, v=v)
    assert info["steps_done"] == 2
    _check(ctx, w, d, ps, u, v, info, True)
    kept = [1.0, 1.25, 1.5]
    u, v, info = api.sa_scale(ctx, d, kept, 1e-6, 20000, kernel="step", warm_keep_v=True)
    _check(ctx, w, d, kept, u, v, info, True)
    # p times 64: references from the row maxima, not from the scaled potentials
    u, v, info = api.sa_scale(ctx, d, [1.0, 64.0], 1e-6, 20000, kernel="step")
    _check(ctx, w, d, [1.0, 64.0], u, v, info, False)


@pytest.mark.parametrize("steps,cap", [(64, 100), (65, 100), (2, 1 << 30)])
def test_resident_limits(ctx, steps, cap):
    """The longest schedule it takes, and calls beyond its parameters (the streaming kernel)."""
    w = W.uniform(100, 1, 1000, 42, dtype=np.int32)
    d = api.to_device(w)
    ps = [1.0 + 0.05 * k for k in range(steps)]
    u, v, info = api.sa_scale(ctx, d, ps, 1e-6, cap, kernel="step")
    assert info["steps_done"] == steps
    _check(ctx, w, d, ps, u, v, info, True)


@pytest.mark.parametrize("kernel,n", [("step", 300), ("step", 3500), ("newton", 300)])
def test_weights_up_to_2_31(ctx, kernel, n):
    """int32 weights over their whole range, on both sides of the log2 table's line (2^15) and
    beyond 24 bits, where a weight is a float and a remainder."""
    rng = np.random.default_rng(44)
    w = np.floor(2.0 ** rng.uniform(13.0, 31.0, (n, n))).astype(np.int64).clip(1, 2 ** 31 - 1).astype(np.int32)
    w[:, :4] = [32767, 32768, 2 ** 24 + 1, 2 ** 31 - 1]
    d = api.to_device(w)
    ps = [1.0, 2.0, 4.0, 8.0]
    u, v, info = api.sa_scale(ctx, d, ps, 1e-6, 20000, kernel=kernel)
    assert info["status"] == 0, info
    assert max(api.sa_verify(ctx, d, ps[-1], u, v)) < SUM_BOUND


def _launches(call):
    """The call's result and the kernels it launched: from a cold start the resident kernel
    is one launch, the streaming kernel three (its potentials are converted afterwards)."""
    n0 = L.lib().sa_kernel_launches()
    r = call()
    return r, L.lib().sa_kernel_launches() - n0


# a form of each width with rows of the stripe in shared memory: 19 and 20 rows on 128 and 256
# threads (16 in registers), 20 and 16 on 512 threads (14 in registers, so that the last group
# of eight register rows is partly empty)
@pytest.mark.parametrize("n,grid", [(300, 16), (1000, 52), (1300, 66), (2000, 126)])
def test_resident_rows_in_shared_memory(ctx, n, grid):
    w = W.uniform(n, 1, 1000, 45 + n, dtype=np.int16)
    w[::3, 1::7] = 0
    d = api.to_device(w)
    ps = [1.0, 2.0, 4.0]
    api.sa_set_option(ctx, "max_grid", grid)
    try:
        (u, v, info), k = _launches(lambda: api.sa_scale(ctx, d, ps, 1e-6, 20000, kernel="step"))
    finally:
        api.sa_set_option(ctx, "max_grid", 0)
    assert k == 1
    _check(ctx, w, d, ps, u, v, info, True)


@pytest.mark.parametrize("n", [300, 1300, 3000])
def test_resident_row_sum_out_of_range_ends_every_block(ctx, n):
    """A warm start whose potential of one row is far too large: that row of K underflows, its block
    finds the sum out of range in the middle of a sweep and the others, waiting for its words, leave
    on the error.  The warm start stays as given and the context usable."""
    w = W.uniform(n, 1, 1000, 46, dtype=np.int16)
    d = api.to_device(w)
    ps = [1.0, 2.0]
    u, v, _ = api.sa_scale(ctx, d, ps[:1], 1e-6, 20000, kernel="step")
    for row in (0, n // 3, n - 1) * 3:
        u1, v1 = u.clone(), v.clone()
        u1[row] += 400.0
        u0, v0 = u1.clone(), v1.clone()
        with pytest.raises(api.SaError) as e:
            api.sa_scale(ctx, d, ps, 1e-6, 20000, kernel="step", resume_from=1, u=u1, v=v1)
        assert e.value.status == L.SA_E_NONFINITE, e.value
        assert torch.equal(u1, u0) and torch.equal(v1, v0)
    u, v, info = api.sa_scale(ctx, d, ps, 1e-6, 20000, kernel="step", resume_from=1, u=u, v=v)
    _check(ctx, w, d, ps, u, v, info, n <= 1300)


def test_resident_subnormal_column_sums(ctx):
    """A column whose entries of K lie at 2^-125.6: in the first sweep its sum is 2^-126.9, below the
    normal FP32 numbers, and its factor 2^126.9 is still finite.  Two sweeps against the same two in
    FP64; FP32 keeps 19 bits of the column's terms, a wrong exponent would be off by 0.3 or more."""
    n, p = 16, 6.28
    w = np.full((n, n), 1 << 20, dtype=np.int32)
    w[:, 0] = 0
    w[:6, 0] = 1
    u, v, info = api.sa_scale(ctx, api.to_device(w), [p], 1e-12, 2, kernel="step")
    assert info["sweeps_total"] == 2, info
    b = p * oracle.log_weights(w.astype(np.int64))
    vo = np.zeros(n)
    for _ in range(2):
        uo = np.log(np.exp(b - vo - 80.0).sum(1)) + 80.0
        vo = np.log(np.exp(b - uo[:, None]).sum(0))
    assert np.max(np.abs(v.cpu().numpy() - vo)) < 1e-3
    assert np.max(np.abs(u.cpu().numpy() - uo)) < 1e-3
    # three entries: the sum is 2^-128 and the factor beyond 2^127 is cut, not infinite
    w[3:6, 0] = 0
    u, v, info = api.sa_scale(ctx, api.to_device(w), [p], 1e-12, 2, kernel="step")
    assert info["status"] == L.SA_E_NOT_CONVERGED, info
    assert torch.isfinite(u).all() and torch.isfinite(v).all()


@pytest.mark.parametrize("n", [130, 600, 1500, 2500])
def test_streaming_forms_below_the_resident_range(ctx, n):
    """The streaming kernel at sizes the resident one usually takes (every width below 4096), reached by
    a schedule longer than the resident kernel's 64 steps."""
    w = W.uniform(n, 1, 1000, 47, dtype=np.int16)
    d = api.to_device(w)
    ps = [1.0 + 0.05 * k for k in range(65)]
    (u, v, info), k = _launches(lambda: api.sa_scale(ctx, d, ps, 1e-6, 20000, kernel="step"))
    assert k == 3 and info["steps_done"] == 65
    _check(ctx, w, d, ps, u, v, info, False)
    b = oracle.log_weights(w.astype(np.int64))
    uo, vo, _, _, st = oracle.sinkhorn(b, ps[-1:], 1e-6, 20000)
    assert st == 0
    x, xo = (oracle.xmatrix(b, ps[-1], *uv) for uv in ((u.cpu().numpy(), v.cpu().numpy()), (uo, vo)))
    assert np.all(np.abs(x - xo) <= 8e-6 * np.maximum(xo, 1.0 / n) + 1e-9)


@pytest.mark.parametrize("n", [1, 300, 1216, 2047, 3333])
def test_which_sizes_are_resident(ctx, n):
    d = api.to_device(W.uniform(n, 1, 1000, 48, dtype=np.int16))
    assert _launches(lambda: api.sa_scale(ctx, d, [1.0], 1e-6, 20000, kernel="step"))[1] == 1


def test_which_sizes_are_streamed(ctx):
    d = api.to_device(W.uniform(3501, 1, 1000, 48, dtype=np.int16))
    assert _launches(lambda: api.sa_scale(ctx, d, [1.0], 1e-6, 20000, kernel="step"))[1] == 3
