// prune.cu -- reduced instance B (Eq. matrixred) as CSR, the certificate of Prop. aoc,
// the LP-duality check of a solution on all of A, and int32 -> int16 narrowing.
//
// Keep test: x_ij(p) >= t  <=>  E_ij = p log2 w_ij - U_i - V_j >= log2 t  (log2 units).
// E is first evaluated in FP32 with the same centring as the sweeps; when it lies within
// a margin of the threshold (a bound on the FP32 error, 1e-4 + 4e-6 p) the decision is
// taken again in FP64, so every decision equals the FP64 one (up to the last bit of the
// FP64 logarithm).  Row and column guards (largest entry of every row and column) use the
// FP32 values with the lowest index on ties.
//
// One read of the matrix screens every entry (prune_scan_kernel): it leaves a bit per
// kept entry, the rows' counts and the largest entry of every row and column; the guards
// then set their bits, and the CSR is written from the bits (n^2 / 8 bytes) and the kept
// weights alone, columns ascending.  Reading the matrix three times with 2-byte loads, once
// for the rows, once for the columns and once to write, took 148 + 265 + 337 us at n = 8192
// (int16, 74 kept entries a row); the scan takes 102 us, bound by its instructions (about 20 an
// entry), the write 16 us.
// This file is compiled without FMA contraction so that the keep predicate evaluates to
// the same value wherever it stands.
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "sa_internal.h"

namespace sa {
namespace {

constexpr int kScanThreads = 256;
constexpr int kScanWarps = kScanThreads / 32;
constexpr int kScanVec = 8;                    // columns of a lane: a byte of keep bits
constexpr int kScanTile = 32 * kScanVec;       // columns of a warp
constexpr int kScanRows = 4;                   // rows whose loads are issued together

struct PruneView {
    const void* w;
    int i16;
    int n;
    int64_t ld;
    double p;
    float pf;
    const double* U;    // log2 units, FP64
    const double* V;
    const float* Lr;    // float(U / p)
    const float* Dr;    // U - p*Lr
    const float* Vf;    // float(V)
    const float* Vd;    // V - Vf
    double log2t;
    float log2tf;
    float margin;
};

__device__ __forceinline__ int load_w(const PruneView& P, int i, int j) {
    return P.i16 ? (int)((const int16_t*)P.w)[(int64_t)i * P.ld + j]
                 : ((const int32_t*)P.w)[(int64_t)i * P.ld + j];
}

// FP32 screened value of E_ij (log2 units)
__device__ __forceinline__ float e32(float pf, float lr, float dr, float vf, float vd, int w) {
    const float L = lg2_approx((float)w);
    return fmaf(pf, L - lr, -vf) - (dr + vd);
}

// the FP64 decision of an entry whose FP32 value lies within the margin of the threshold (or
// is not a number); not inlined: it is rare, and the scan's loop is unrolled 32 times
__device__ __noinline__ bool keep_near(const PruneView& P, int i, int j, int w) {
    const double ed = (w > 0 ? P.p * log2((double)w) : -INFINITY) - P.U[i] - P.V[j];
    return ed >= P.log2t;
}

// The eight weights of a row at column j0 (cnt of them inside the matrix, zeros after) as
// they lie in memory: 16-byte loads where the rows start on 16-byte boundaries.
template <typename WT>
struct Raw8 {
    uint4 q[8 * sizeof(WT) / 16];
    __device__ __forceinline__ void load(const void* w, int64_t ld, int vec_ok, int row, int j0, int cnt) {
        const WT* src = (const WT*)w + (int64_t)row * ld + j0;
        if (vec_ok && cnt == kScanVec) {
#pragma unroll
            for (int h = 0; h < (int)(sizeof(q) / 16); ++h) q[h] = __ldg((const uint4*)src + h);
        } else {
            unsigned o[sizeof(q) / 4];
#pragma unroll
            for (int h = 0; h < (int)(sizeof(q) / 4); ++h) {
                const int per = 4 / sizeof(WT), e = h * per;
                o[h] = e < cnt ? (unsigned)src[e] & (sizeof(WT) == 2 ? 0xffffu : 0xffffffffu) : 0u;
                if (sizeof(WT) == 2 && e + 1 < cnt) o[h] |= (unsigned)src[e + 1] << 16;
            }
#pragma unroll
            for (int h = 0; h < (int)(sizeof(q) / 16); ++h) q[h] = make_uint4(o[4 * h], o[4 * h + 1], o[4 * h + 2], o[4 * h + 3]);
        }
    }
    __device__ __forceinline__ unsigned word(int h) const {
        const uint4& v = q[h >> 2];
        return (h & 3) == 0 ? v.x : (h & 3) == 1 ? v.y : (h & 3) == 2 ? v.z : v.w;
    }
    __device__ __forceinline__ int get(int e) const {
        if (sizeof(WT) == 4) return (int)word(e);
        return (e & 1) ? (int)word(e >> 1) >> 16 : (int)(short)(word(e >> 1) & 0xffffu);
    }
};

// Rows a warp of the scan kernels takes: a few waves of blocks where the matrix has them, at
// least one group of rows and at most 32.
int scan_rows_per_warp(const sa_ctx* ctx, int n) {
    const int tiles = (n + kScanTile - 1) / kScanTile;
    const int want = std::max(1, 16 * ctx->num_sms / tiles) * kScanWarps;
    const int r = (int)align_up((size_t)(n + want - 1) / want, kScanRows);
    return std::min(32, std::max(kScanRows, r));
}

// (value, index) as a key whose maximum is the largest value and, on ties, the lowest index.
// A NaN counts as no entry.
__device__ __forceinline__ unsigned order_key(float e) {
    const unsigned b = __float_as_uint(e + 0.0f);   // -0 ties with +0
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ unsigned long long arg_key(unsigned key, int idx) {
    return ((unsigned long long)key << 32) | (0xffffffffu - (unsigned)idx);
}
__device__ __forceinline__ int key_index(unsigned long long k) { return (int)(0xffffffffu - (unsigned)k); }

// One read of the matrix.  A warp owns a tile of 256 columns, eight a lane, and rpw rows;
// the eight warps of a block take consecutive row chunks of one tile, so that a block has
// one candidate per column.  Per row the warp adds its count and its largest entry to the
// row's, per tile the block its largest entries to the columns' (integer atomics: the result
// does not depend on their order).
template <typename WT>
__global__ void __launch_bounds__(kScanThreads) prune_scan_kernel(PruneView P, int vec_ok, int rpw, int* cnt,
                                                                  unsigned long long* rkey, unsigned long long* ckey,
                                                                  unsigned char* mask, int pitch) {
    __shared__ unsigned long long sk[kScanWarps][kScanTile];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int n = P.n;
    const int j0 = blockIdx.x * kScanTile + lane * kScanVec;
    const int nv = max(0, min(kScanVec, n - j0));
    const int r0 = (blockIdx.y * kScanWarps + wid) * rpw, r1 = min(n, r0 + rpw);
    float vf[kScanVec], vd[kScanVec], cbest[kScanVec];
    int crow[kScanVec];
#pragma unroll
    for (int e = 0; e < kScanVec; ++e) {
        vf[e] = e < nv ? P.Vf[j0 + e] : 0.0f;
        vd[e] = e < nv ? P.Vd[j0 + e] : 0.0f;
        cbest[e] = -INFINITY;
        crow[e] = r0;
    }
    for (int rb = r0; rb < r1; rb += kScanRows) {
        Raw8<WT> w[kScanRows];
#pragma unroll
        for (int r = 0; r < kScanRows; ++r) w[r].load(P.w, P.ld, vec_ok, min(rb + r, r1 - 1), j0, nv);
#pragma unroll
        for (int r = 0; r < kScanRows; ++r) {
            const int i = rb + r;
            if (i >= r1) break;
            const float lr = P.Lr[i], dr = P.Dr[i];
            unsigned bits = 0, near = 0;
            float best = -INFINITY;
            float x[kScanVec];
#pragma unroll
            for (int e = 0; e < kScanVec; ++e) {   // lanes past the matrix hold zero weights
                const int wv = w[r].get(e);
                x[e] = wv > 0 ? e32(P.pf, lr, dr, vf[e], vd[e], wv) : -INFINITY;
                bits |= (x[e] >= P.log2tf ? 1u : 0u) << e;
                near |= (fabsf(x[e] - P.log2tf) > P.margin ? 0u : 1u) << e;
                best = fmaxf(best, x[e]);          // drops NaN, as the comparison below does
                if (x[e] > cbest[e]) { cbest[e] = x[e]; crow[e] = i; }
            }
            for (near &= (1u << nv) - 1u; near; near &= near - 1) {
                const int e = __ffs(near) - 1;
                int wv = 0;
#pragma unroll
                for (int h = 0; h < kScanVec; ++h) wv = h == e ? w[r].get(h) : wv;
                bits = (bits & ~(1u << e)) | ((keep_near(P, i, j0 + e, wv) ? 1u : 0u) << e);
            }
            __syncwarp();
            int bj = j0;
#pragma unroll
            for (int e = kScanVec - 1; e >= 0; --e) bj = x[e] == best ? j0 + e : bj;   // the lowest
            if (!(best > -INFINITY)) bj = j0;
            mask[(size_t)i * pitch + (j0 >> 3)] = (unsigned char)bits;
            const int c = __reduce_add_sync(0xffffffffu, __popc(bits));
            const unsigned key = order_key(best);
            const unsigned top = __reduce_max_sync(0xffffffffu, key);
            const int src = __ffs(__ballot_sync(0xffffffffu, key == top)) - 1;   // lanes ascend in j
            if (lane == src) atomicMax(rkey + i, arg_key(key, bj));
            if (lane == 0 && c > 0) atomicAdd(cnt + i, c);
        }
    }
#pragma unroll
    for (int e = 0; e < kScanVec; ++e) sk[wid][lane * kScanVec + e] = r0 < r1 ? arg_key(order_key(cbest[e]), crow[e]) : 0ull;
    __syncthreads();
    const int c = threadIdx.x, j = blockIdx.x * kScanTile + c;
    static_assert(kScanThreads == kScanTile, "a thread per column of the tile");
    unsigned long long k = 0ull;
#pragma unroll
    for (int x = 0; x < kScanWarps; ++x) k = max(k, sk[x][c]);
    if (j < n) atomicMax(ckey + j, k);
}

// The certificate terms max_j (p ln w_ij - v_j) of the rows, evaluated in FP64 at the
// largest entry, and with guard != 0 the bits of the largest entry of every row and column
// (counted where the bit was not yet set).
__global__ void guard_kernel(PruneView P, int guard, const unsigned long long* rkey, const unsigned long long* ckey, int* cnt,
                             unsigned* mask, int pitch_words, double* rterm) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= 2 * P.n) return;
    int i, j;
    if (k < P.n) {
        i = k;
        j = key_index(rkey[k]);
        const int w = load_w(P, i, j);
        rterm[i] = (w > 0 ? P.p * log((double)w) : -INFINITY) - P.V[j] * kLn2;
    } else {
        j = k - P.n;
        i = key_index(ckey[j]);
    }
    if (!guard) return;
    const unsigned bit = 1u << (j & 31);
    if (!(atomicOr(mask + (size_t)i * pitch_words + (j >> 5), bit) & bit)) atomicAdd(cnt + i, 1);
}

// Exclusive scan of n counts into row_ptr[0..n] (single block, n any size): each thread sums
// a run of consecutive counts, one block scan of the runs' sums.
__global__ void __launch_bounds__(1024) scan_kernel(const int* cnt, int64_t* row_ptr, int n) {
    __shared__ int64_t sh[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int per = (n + 1023) / 1024;
    const int i0 = min(n, (int)threadIdx.x * per), i1 = min(n, i0 + per);
    int64_t v = 0;
    for (int i = i0; i < i1; ++i) v += cnt[i];
    int64_t s = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += y;
    }
    if (lane == 31) sh[wid] = s;
    __syncthreads();
    int64_t at = s - v;
#pragma unroll
    for (int x = 0; x < 32; ++x) at += x < wid ? sh[x] : 0;
    for (int i = i0; i < i1; ++i) {
        row_ptr[i] = at;
        at += cnt[i];
    }
    if (threadIdx.x == 1023) row_ptr[n] = at;
}

// The kept columns and weights of each row in ascending order, from the keep bits: a warp
// per row, 32 words (1024 columns) at a time.
__global__ void __launch_bounds__(256) prune_write_kernel(PruneView P, const unsigned* mask, int pitch_words,
                                                          const int64_t* row_ptr, int32_t* col, int32_t* wout) {
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (i >= P.n) return;
    int64_t pos = row_ptr[i];
    const int words = (P.n + 31) / 32;
    for (int b = 0; b < words; b += 32) {
        unsigned m = b + lane < words ? mask[(size_t)i * pitch_words + b + lane] : 0u;
        const int c = __popc(m);
        int s = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        int64_t at = pos + s - c;
        while (m) {
            const int j = 32 * (b + lane) + __ffs(m) - 1;
            col[at] = j;
            wout[at] = load_w(P, i, j);
            ++at;
            m &= m - 1;
        }
        pos += __shfl_sync(0xffffffffu, s, 31);
    }
}

__global__ void prune_prep_kernel(const double* u, const double* v, int n, double p, double* U,
                                  double* V, float* Lr, float* Dr, float* Vf, float* Vd, int* cnt,
                                  unsigned long long* rkey, unsigned long long* ckey) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    cnt[k] = 0;
    rkey[k] = ckey[k] = 0ull;
    const double uu = u[k] * kLog2e, vv = v[k] * kLog2e;
    U[k] = uu;
    V[k] = vv;
    const float lr = (float)(uu / p);
    Lr[k] = lr;
    Dr[k] = (float)(uu - p * (double)lr);
    const float vf = (float)vv;
    Vf[k] = vf;
    Vd[k] = (float)(vv - (double)vf);
}

// ---- certificate check on all of A --------------------------------------------------
struct CertView {
    const void* w;
    int n;
    int64_t ld;
    int vec_ok;
    const double* alpha;
    const double* beta;
    const float* af;
    const float* bf;
    double tau;
};

// alpha and beta (consecutive) in FP32; clears the counter
__global__ void cert_prep_kernel(const double* x, float* y, int n, unsigned long long* count) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) y[k] = (float)x[k];
    if (k == 0) *count = 0ull;
}

// log w - alpha - beta in FP64; not inlined, as keep_near
__device__ __noinline__ double dual_gap(const CertView& C, int i, int j, int w) {
    return log((double)w) - C.alpha[i] - C.beta[j];
}

// One read of the matrix, bound by it: warps on tiles of 256 columns with 16-byte loads of
// four rows in flight, as in prune_scan_kernel: 28 us at n = 5001, int32 (3.6 TB/s), where a
// block per row with one 4-byte load in flight a thread took 45 us.
template <typename WT>
__global__ void __launch_bounds__(kScanThreads) certify_kernel(CertView C, int rpw, unsigned long long* count, int64_t max_add,
                                                               int3* add) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int n = C.n;
    const int j0 = blockIdx.x * kScanTile + lane * kScanVec;
    const int nv = max(0, min(kScanVec, n - j0));
    const int r0 = (blockIdx.y * kScanWarps + wid) * rpw, r1 = min(n, r0 + rpw);
    if (nv == 0) return;
    float bf[kScanVec];
#pragma unroll
    for (int e = 0; e < kScanVec; ++e) bf[e] = e < nv ? C.bf[j0 + e] : 0.0f;
    for (int rb = r0; rb < r1; rb += kScanRows) {
        Raw8<WT> w[kScanRows];
#pragma unroll
        for (int r = 0; r < kScanRows; ++r) w[r].load(C.w, C.ld, C.vec_ok, min(rb + r, r1 - 1), j0, nv);
#pragma unroll
        for (int r = 0; r < kScanRows; ++r) {
            const int i = rb + r;
            if (i >= r1) break;
            const float af = C.af[i];
            unsigned near = 0;
#pragma unroll
            for (int e = 0; e < kScanVec; ++e) {
                const int wv = w[r].get(e);
                const float g = lg2_approx((float)wv) * (float)kLn2 - af - bf[e];
                // FP32 error of g is below 1e-5 for |alpha|, |beta| < 1e3; re-check in FP64 near tau
                near |= (wv <= 0 || g < (float)C.tau - 1e-4f ? 0u : 1u) << e;
            }
            for (; near; near &= near - 1) {
                const int e = __ffs(near) - 1;
                int wv = 0;
#pragma unroll
                for (int h = 0; h < kScanVec; ++h) wv = h == e ? w[r].get(h) : wv;
                if (dual_gap(C, i, j0 + e, wv) > C.tau) {
                    const unsigned long long k = atomicAdd(count, 1ull);
                    if ((int64_t)k < max_add) add[k] = make_int3(i, j0 + e, wv);
                }
            }
        }
    }
}

// smallest positive and largest weight of the matrix (zeros are absent entries)
__global__ void minmax_kernel(const void* w, int i16, int n, int64_t ld, unsigned long long* out) {
    unsigned mn = 0xffffffffu, mx = 0u;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (int64_t)n * n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / n), j = (int)(e % n);
        const int x = i16 ? (int)((const int16_t*)w)[(int64_t)i * ld + j] : ((const int32_t*)w)[(int64_t)i * ld + j];
        if (x > 0) {
            mn = min(mn, (unsigned)x);
            mx = max(mx, (unsigned)x);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMin(out, (unsigned long long)mn);
        atomicMax(out + 1, (unsigned long long)mx);
    }
}

__global__ void narrow_kernel(const int32_t* src, int64_t lds, int16_t* dst, int64_t ldd, int n,
                              unsigned long long* bad) {
    const int i = blockIdx.y;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        int v = src[(int64_t)i * lds + j];
        if (v < 0 || v > 32767) {
            atomicAdd(bad, 1ull);
            v = v < 0 ? 0 : 32767;
        }
        dst[(int64_t)i * ldd + j] = (int16_t)v;
    }
}

}  // namespace

// rows start on 16-byte boundaries
static int rows_aligned(const sa_matrix* a) {
    return ((uintptr_t)a->w & 15) == 0 && ((size_t)a->ld * wbytes(a->wtype)) % 16 == 0;
}

// entries a row of the CSR that prune_device keeps room for in the workspace
constexpr int64_t kCsrPerRow = 128;

sa_status prune_device(sa_ctx* ctx, const sa_matrix* a, double p, const double* d_u,
                       const double* d_v, double t, int guard, sa_csr* out, double* log_ub) {
    const int n = a->n;
    cudaStream_t st = ctx->stream;
    if (!(t > 0)) t = 1.0 / n;
    const int tiles = (n + kScanTile - 1) / kScanTile;
    const int pitch = tiles * kScanVec * 4;   // bytes of keep bits a row
    const size_t fixed = 5 * align_up((size_t)n * 8, 256) + 5 * align_up((size_t)n * 4, 256) +
                         align_up((size_t)(n + 1) * 8, 256) + align_up((size_t)n * pitch, 256) + 4096;
    const size_t room = (size_t)std::min<int64_t>((int64_t)n * n, kCsrPerRow * n);
    sa_status rc = ctx->ws.reserve(fixed + 2 * align_up(room * 4, 256));
    if (rc) return rc;
    // pinned: row_ptr, the certificate terms of the rows, v
    rc = ctx->pinned.reserve((size_t)(3 * (int64_t)n + 1) * 8);
    if (rc) return rc;
    int64_t* h_rp = (int64_t*)ctx->pinned.ptr;
    double* h_rterm = (double*)(h_rp + n + 1);
    double* h_v = h_rterm + n;
    Carve cv(ctx->ws.ptr);
    double* U = cv.take<double>(n);
    double* V = cv.take<double>(n);
    float* Lr = cv.take<float>(n);
    float* Dr = cv.take<float>(n);
    float* Vf = cv.take<float>(n);
    float* Vd = cv.take<float>(n);
    int* cnt = cv.take<int>(n);
    unsigned long long* rkey = cv.take<unsigned long long>(n);
    unsigned long long* ckey = cv.take<unsigned long long>(n);
    double* rterm = cv.take<double>(n);
    int64_t* row_ptr = cv.take<int64_t>(n + 1);
    unsigned* mask = cv.take<unsigned>((size_t)n * pitch / 4);
    prune_prep_kernel<<<(n + 255) / 256, 256, 0, st>>>(d_u, d_v, n, p, U, V, Lr, Dr, Vf, Vd, cnt, rkey, ckey);
    PruneView P;
    P.w = a->w;
    P.i16 = a->wtype == SA_I16;
    P.n = n;
    P.ld = a->ld;
    P.p = p;
    P.pf = (float)p;
    P.U = U;
    P.V = V;
    P.Lr = Lr;
    P.Dr = Dr;
    P.Vf = Vf;
    P.Vd = Vd;
    P.log2t = std::log2(t);
    P.log2tf = (float)P.log2t;
    P.margin = (float)(1e-4 + 4e-6 * p);
    const int rpw = scan_rows_per_warp(ctx, n);
    const dim3 g(tiles, (n + rpw * kScanWarps - 1) / (rpw * kScanWarps));
    if (P.i16) prune_scan_kernel<int16_t><<<g, kScanThreads, 0, st>>>(P, rows_aligned(a), rpw, cnt, rkey, ckey, (unsigned char*)mask, pitch);
    else prune_scan_kernel<int32_t><<<g, kScanThreads, 0, st>>>(P, rows_aligned(a), rpw, cnt, rkey, ckey, (unsigned char*)mask, pitch);
    guard_kernel<<<(2 * n + 255) / 256, 256, 0, st>>>(P, guard, rkey, ckey, cnt, mask, pitch / 4, rterm);
    scan_kernel<<<1, 1024, 0, st>>>(cnt, row_ptr, n);
    count_launch(4);
    SA_CUDA(cudaMemcpyAsync(h_rp, row_ptr, (size_t)(n + 1) * 8, cudaMemcpyDeviceToHost, st));
    SA_CUDA(cudaMemcpyAsync(h_rterm, rterm, (size_t)n * 8, cudaMemcpyDeviceToHost, st));
    SA_CUDA(cudaMemcpyAsync(h_v, d_v, (size_t)n * 8, cudaMemcpyDeviceToHost, st));
    SA_CUDA(cudaStreamSynchronize(st));
    SA_CUDA(cudaGetLastError());
    const int64_t nnz = h_rp[n];
    // the device CSR: behind the vectors in the workspace where it fits (after a scaling of
    // the same matrix it always does), else for the call alone
    const size_t entries = (size_t)std::max<int64_t>(nnz, 1);
    int32_t* own = nullptr;
    int32_t *d_col, *d_w;
    if (align_up(cv.off, 256) + 2 * align_up(entries * 4, 256) <= ctx->ws.size) {
        d_col = cv.take<int32_t>(entries);
        d_w = cv.take<int32_t>(entries);
    } else {
        SA_CUDA(cudaMallocAsync((void**)&own, 2 * entries * 4, st));
        d_col = own;
        d_w = own + entries;
    }
    prune_write_kernel<<<(n + 7) / 8, 256, 0, st>>>(P, mask, pitch / 4, row_ptr, d_col, d_w);
    count_launch();
    rc = csr_alloc(out, n, nnz);
    if (rc) {
        if (own) cudaFreeAsync(own, st);
        return rc;
    }
    SA_CUDA(cudaMemcpyAsync(out->col, d_col, (size_t)nnz * 4, cudaMemcpyDeviceToHost, st));
    SA_CUDA(cudaMemcpyAsync(out->w, d_w, (size_t)nnz * 4, cudaMemcpyDeviceToHost, st));
    if (own) SA_CUDA(cudaFreeAsync(own, st));
    std::copy(h_rp, h_rp + n + 1, out->row_ptr);
    if (log_ub) {
        double acc = 0.0;
        for (int i = 0; i < n; ++i) acc += h_rterm[i];
        for (int j = 0; j < n; ++j) acc += h_v[j];
        *log_ub = acc / p;
    }
    SA_CUDA(cudaStreamSynchronize(st));
    SA_CUDA(cudaGetLastError());
    return SA_OK;
}

// additions that come back with the count in one copy
constexpr int64_t kCertFirst = 2048;

sa_status certify_device(sa_ctx* ctx, const sa_matrix* a, const double* alpha, const double* beta,
                         double tau, int64_t* n_viol, int64_t max_add, sa_csr* add) {
    const int n = a->n;
    cudaStream_t st = ctx->stream;
    if (max_add < 0) max_add = 0;
    const size_t list_bytes = 16 + sizeof(int3) * (size_t)std::max<int64_t>(max_add, 1);
    sa_status rc = ctx->ws.reserve(align_up((size_t)2 * n * 8, 256) + align_up((size_t)2 * n * 4, 256) +
                                   align_up(list_bytes, 256) + 1024);
    if (rc) return rc;
    const size_t first_bytes = 16 + sizeof(int3) * (size_t)(add ? std::min(max_add, kCertFirst) : 0);
    rc = ctx->pinned.reserve((size_t)2 * n * 8 + first_bytes);
    if (rc) return rc;
    double* h_ab = (double*)ctx->pinned.ptr;
    const unsigned char* h_list = (const unsigned char*)(h_ab + 2 * (size_t)n);
    std::copy(alpha, alpha + n, h_ab);
    std::copy(beta, beta + n, h_ab + n);
    Carve cv(ctx->ws.ptr);
    double* ab = cv.take<double>(2 * (size_t)n);
    float* abf = cv.take<float>(2 * (size_t)n);
    unsigned char* list = cv.take<unsigned char>(list_bytes);   // the count, then the additions
    unsigned long long* count = (unsigned long long*)list;
    int3* adds = (int3*)(list + 16);
    SA_CUDA(cudaMemcpyAsync(ab, h_ab, (size_t)2 * n * 8, cudaMemcpyHostToDevice, st));
    cert_prep_kernel<<<(2 * n + 255) / 256, 256, 0, st>>>(ab, abf, 2 * n, count);
    const CertView C{a->w, n, a->ld, rows_aligned(a), ab, ab + n, abf, abf + n, tau};
    const int rpw = scan_rows_per_warp(ctx, n);
    const dim3 g((n + kScanTile - 1) / kScanTile, (n + rpw * kScanWarps - 1) / (rpw * kScanWarps));
    if (a->wtype == SA_I16) certify_kernel<int16_t><<<g, kScanThreads, 0, st>>>(C, rpw, count, max_add, adds);
    else certify_kernel<int32_t><<<g, kScanThreads, 0, st>>>(C, rpw, count, max_add, adds);
    count_launch(2);
    SA_CUDA(cudaMemcpyAsync((void*)h_list, list, first_bytes, cudaMemcpyDeviceToHost, st));
    SA_CUDA(cudaStreamSynchronize(st));
    SA_CUDA(cudaGetLastError());
    const int64_t h_count = (int64_t)*(const unsigned long long*)h_list;
    *n_viol = h_count;
    if (add) {
        const int64_t k = std::min<int64_t>(h_count, max_add);
        std::vector<int3> list_h(k);
        const int64_t have = std::min(k, kCertFirst);
        std::copy((const int3*)(h_list + 16), (const int3*)(h_list + 16) + have, list_h.begin());
        if (k > have) {
            SA_CUDA(cudaMemcpyAsync(list_h.data() + have, adds + have, (size_t)(k - have) * sizeof(int3), cudaMemcpyDeviceToHost, st));
            SA_CUDA(cudaStreamSynchronize(st));
        }
        std::sort(list_h.begin(), list_h.end(), [](const int3& x, const int3& y) { return x.x != y.x ? x.x < y.x : x.y < y.y; });
        rc = csr_alloc(add, n, k);
        if (rc) return rc;
        std::fill(add->row_ptr, add->row_ptr + n + 1, 0);
        for (int64_t x = 0; x < k; ++x) {
            add->row_ptr[list_h[x].x + 1]++;
            add->col[x] = list_h[x].y;
            add->w[x] = list_h[x].z;
        }
        for (int r = 0; r < n; ++r) add->row_ptr[r + 1] += add->row_ptr[r];
    }
    return SA_OK;
}

sa_status weights_minmax(sa_ctx* ctx, const sa_matrix* a, int64_t* wmin, int64_t* wmax) {
    cudaStream_t st = ctx->stream;
    sa_status rc = ctx->ws.reserve(256);
    if (rc) return rc;
    unsigned long long* d = (unsigned long long*)ctx->ws.ptr;
    const unsigned long long init[2] = {~0ull, 0ull};
    SA_CUDA(cudaMemcpyAsync(d, init, sizeof(init), cudaMemcpyHostToDevice, st));
    const int64_t total = (int64_t)a->n * a->n;
    const int blocks = (int)std::min<int64_t>((total + 255) / 256, (int64_t)ctx->num_sms * 8);
    minmax_kernel<<<blocks, 256, 0, st>>>(a->w, a->wtype == SA_I16, a->n, a->ld, d);
    count_launch();
    unsigned long long h[2];
    SA_CUDA(cudaMemcpyAsync(h, d, sizeof(h), cudaMemcpyDeviceToHost, st));
    SA_CUDA(cudaStreamSynchronize(st));
    if (h[1] == 0ull) { set_error("matrix has no positive entry"); return SA_E_NO_PERFECT_MATCHING; }
    *wmin = (int64_t)h[0];
    *wmax = (int64_t)h[1];
    return SA_OK;
}

sa_status narrow_device(sa_ctx* ctx, const int32_t* src, int64_t lds, int16_t* dst, int64_t ldd,
                        int n, int64_t* n_bad) {
    cudaStream_t st = ctx->stream;
    sa_status rc = ctx->ws.reserve(256);
    if (rc) return rc;
    unsigned long long* bad = (unsigned long long*)ctx->ws.ptr;
    SA_CUDA(cudaMemsetAsync(bad, 0, 8, st));
    dim3 g((n + 255) / 256 < 8 ? (n + 255) / 256 : 8, n);
    narrow_kernel<<<g, 256, 0, st>>>(src, lds, dst, ldd, n, bad);
    count_launch();
    unsigned long long h = 0;
    SA_CUDA(cudaMemcpyAsync(&h, bad, 8, cudaMemcpyDeviceToHost, st));
    SA_CUDA(cudaStreamSynchronize(st));
    SA_CUDA(cudaGetLastError());
    if (n_bad) *n_bad = (int64_t)h;
    return SA_OK;
}

}  // namespace sa
