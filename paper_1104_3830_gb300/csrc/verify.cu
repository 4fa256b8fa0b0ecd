// verify.cu -- FP64 row and column sums of X(p) from the potentials (sa_verify), one read of
// the matrix for both.
//
// What bounds it: GB300 runs two FP64 instructions per clock and SM, so the FP64 exp and log
// of every entry (about 55 instructions), taken once for the rows and once for the columns,
// cost 12.7 ms at n = 8192 against 20 us for the bytes.  Here the exponent
//     E_ij = p log2 w_ij - U_i - V_j            (U = u log2 e, V = v log2 e)
// is formed exactly in 64-bit fixed point (integer adds run at 32 times the FP64 rate): the
// weights below 2^15 take p log2 w from a table made per call, a larger weight its top 15
// bits from the table and the rest from the series of log2(1 + d), d < 2^-14.  2^E follows from the
// integer part of E (the exponent field), 12 bits (a 4096-entry table in shared memory) and
// exp(t) - 1 = t + t^2 (1/2 + t/6), |t| < 2^-13, whose second part (below 2^-27) is formed in FP32.
// Five FP64 instructions per entry are left (int16; nine for weights above 2^15), two of them
// the sums: 0.78 - 0.81 ms at n = 8192 (0.57 ms of it those five at the FP64 rate).
//
// Error: the fraction has F = 61 - ceil(log2 M) bits, M the largest of p log2 w, |U| and |V|, and
// the table's logarithms are formed to 2^-57, so E is off by a few 2^-F, where
// exp(p log(w) - u - v) in FP64 rounds the logarithm, the product and both differences at
// their magnitude: against extended precision the sums of n = 1000 matrices at p = 64 .. 512 are
// off by 1e-16 to 1.2e-14 (relative, 2-norm), by 6e-15 to 2e-13 in that formula.  Potentials
// that are not finite or leave F below 44 take that formula instead (mode 0).  The tables pay at
// every size: 59 - 75 us for a call with n = 8 .. 512 (int32), 61 - 171 us with mode 0.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "sa_internal.h"

namespace sa {
namespace {

constexpr int kVerifyThreads = 256;
constexpr int kVerifyWarps = kVerifyThreads / 32;
constexpr int kVerifyGroup = 8;                     // rows reduced together
constexpr int kVerifyTab = 32768;                   // weights with a table entry of p log2 w
constexpr int kExpTab = 4096;

struct VerifyParams {
    int mode;        // 1: fixed point, 0: FP64 exp and log
    int F;           // fraction bits
    long long pfix;  // p in fixed point
    double clog;     // p log2(e) 2^F
};

struct VerifyView {
    const void* w;
    int n;
    int64_t ld;
    int vec_ok;      // rows start on 16-byte boundaries
    double p;
    const double* u;
    const double* v;
    const long long* Uf;
    const long long* Vf;
    const long long* T;    // p log2 w, w < kVerifyTab
    const double* R;       // 1 / w, w < kVerifyTab
    const double* E;       // 2^((k + 1/2) / 4096)
    const VerifyParams* par;
    int rows_per_warp;
    double* rpart;   // [column tiles][n]
    double* cpart;   // [row chunks][n]
};

// One block: the largest magnitude of the potentials and of p log2 w gives F.
__global__ void __launch_bounds__(1024) verify_bounds_kernel(const double* u, const double* v, int n, double p, double log2w_max,
                                     VerifyParams* par) {
    __shared__ double sh[32];
    double m = p * log2w_max;
    int bad = 0;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const double a = fabs(u[k]) * kLog2e, b = fabs(v[k]) * kLog2e;
        if (!(a < INFINITY) || !(b < INFINITY)) bad = 1;
        m = fmax(m, fmax(a, b));
    }
    m = warp_max(m);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) m = fmax(m, sh[k]);
        VerifyParams o{0, 0, 0, 0.0};
        if (!bad && m < 0x1p17) {
            const int F = min(57, 61 - ilogb(m + 1.0) - 1);   // m < 2^(61 - F)
            o.F = F;
            o.mode = F >= 44;
            o.pfix = llrint(ldexp(p, F));
            o.clog = ldexp(p * kLog2e, F);
        }
        *par = o;
    }
}

// x y 2^F rounded to an integer, the product taken exactly
__device__ __forceinline__ long long fixed_product(double x, double y, double ylo, int F) {
    const double h = x * y;
    const double l = fma(x, y, -h) + x * ylo;
    return llrint(ldexp(h, F)) + llrint(ldexp(l, F));
}

// log2 of k (0 < k < 2^15) with 58 fraction bits, digit by digit: the mantissa is squared, and
// each time it passes 2 a bit of the logarithm is 1 (the errors of the truncated squares halve with
// every bit: below 2^-57 in all)
__device__ unsigned long long log2_fixed58(unsigned k) {
    const int e = 31 - __clz(k);
    unsigned long long m = (unsigned long long)k << (63 - e);   // in [1, 2), 63 fraction bits
    unsigned long long f = (unsigned long long)e;
    for (int b = 0; b < 58; ++b) {
        const unsigned long long hi = __umul64hi(m, m), lo = m * m;   // m^2, 126 fraction bits
        if (hi >> 63) {
            m = hi;
            f = 2 * f + 1;
        } else {
            m = (hi << 1) | (lo >> 63);
            f = 2 * f;
        }
    }
    return f;
}

__global__ void verify_tables_kernel(const double* u, const double* v, int n, double p, const VerifyParams* par, long long* Uf,
                                     long long* Vf, long long* T, double* R, double* E) {
    if (!par->mode) return;
    const int F = par->F;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < kVerifyTab) {
        long long t = 0;
        if (k > 0) {
            // p = pm 2^ep with an integer pm < 2^53; pm log2 k 2^58 has at most 115 bits
            const unsigned long long l = log2_fixed58((unsigned)k);
            const int ep = ilogb(p) - 52;
            const unsigned long long pm = (unsigned long long)scalbn(p, -ep);
            const unsigned long long hi = __umul64hi(pm, l), lo = pm * l;
            const int sh = 58 - F - ep;   // > 0: p log2(w) 2^F < 2^61
            if (sh < 64) t = (long long)((hi << (64 - sh)) | (lo >> sh)) + (long long)((lo >> (sh - 1)) & 1u);
            else if (sh == 64) t = (long long)hi + (long long)(lo >> 63);
            else t = sh < 128 ? (long long)(hi >> (sh - 64)) + (long long)((hi >> (sh - 65)) & 1u) : 0;
        }
        T[k] = t;
        R[k] = k > 0 ? 1.0 / (double)k : 0.0;
    }
    if (k < kExpTab) E[k] = exp2((k + 0.5) / kExpTab);
    for (int j = k; j < n; j += gridDim.x * blockDim.x) {
        Uf[j] = fixed_product(u[j], kLog2e, 2.0355273740931033e-17, F);   // log2 e = head + tail
        Vf[j] = fixed_product(v[j], kLog2e, 2.0355273740931033e-17, F);
    }
}

// p log2 w in fixed point
template <typename WT>
__device__ __forceinline__ long long fixed_plog(const VerifyView& A, const VerifyParams& P, int w) {
    if (sizeof(WT) == 2 || w < kVerifyTab) return __ldg(A.T + w);
    const int s = 17 - __clz(w);                       // w >> s in [2^14, 2^15)
    const int hi = w >> s;
    const unsigned lo = (unsigned)w & ((1u << s) - 1u);
    // lo (below 2^17) in FP64 from its FP32 bits (0: 2^-127, which adds nothing)
    const unsigned lb = __float_as_uint((float)(int)lo);
    const double lod = __hiloint2double((int)(lb >> 3) + 0x38000000, (int)(lb << 29));
    const double r = __ldg(A.R + hi);
    const double d = lod * __hiloint2double(__double2hiint(r) - (s << 20), __double2loint(r));   // < 2^-14
    // ln(1 + d) = (d - d^2 / 2) + d^3 (1/3 - d/4): the first part in FP64, the second, below 2^-43, in FP32
    // (d cut to FP32 from its bits; 0: lo = 0, else d is at least 2^-31)
    const float df = lo ? __uint_as_float(((unsigned)(__double2hiint(d) - 0x38000000) << 3) | ((unsigned)__double2loint(d) >> 29)) : 0.0f;
    const unsigned cb = __float_as_uint(df * df * df * (0.333333343f - 0.25f * df));
    const double cd = __hiloint2double((int)(cb >> 3) + 0x38000000, (int)(cb << 29));
    const double nh = __hiloint2double((int)((unsigned)(__double2hiint(d) - 0x100000) ^ 0x80000000u), __double2loint(d));   // -d/2
    // below 2^51: the sum with 1.5 2^52 holds the rounded integer in its low bits
    const double m = fma(P.clog, fma(d, nh, d) + cd, 0x1.8p52);
    return __ldg(A.T + hi) + (long long)s * P.pfix + (__double_as_longlong(m) - 0x4338000000000000ll);
}

// 2^(e 2^-F)
__device__ __forceinline__ double fixed_exp2(long long e, int F, const double* tab) {
    const int k = (int)(e >> F);
    const unsigned long long fr = (unsigned long long)e << (64 - F);
    const double t = tab[(int)(fr >> 52)];
    const long long r = (long long)((fr << 12) ^ 0x8000000000000000ull) >> 12;   // units 2^-64, |r| < 2^51
    const double rd = __longlong_as_double(0x4338000000000000ll + r) - 0x1.8p52;
    const float tf = (float)(int)(r >> 20) * (0.693147182f * 0x1p-44f);
    const float q = tf * tf * (0.5f + tf * 0.166666672f);
    const unsigned qb = __float_as_uint(q);
    const double qd = __hiloint2double((int)(qb >> 3) + 0x38000000, (int)(qb << 29));
    const double y = fma(t, fma(rd, kLn2 * 0x1p-64, qd), t);   // in [1, 2)
    const int hi = __double2hiint(y), lo = __double2loint(y);
    if (k >= -1022 && k <= 1023) return __hiloint2double(hi + (k << 20), lo);
    if (k > 1023) return INFINITY;
    return k < -1080 ? 0.0 : __hiloint2double(hi + ((k + 200) << 20), lo) * 0x1p-200;
}

// A warp owns a tile of 32 VEC columns (VEC = 16 bytes of weights a lane) and rows_per_warp rows;
// the eight warps of a block take consecutive row chunks of one column tile, so that a block
// writes one partial per column.  The row sums of eight rows are reduced together: each
// exchange halves the rows that a lane still carries (9 additions instead of 40).  Three blocks an
// SM (80 registers; the int16 form spills 168 bytes) hide more of the FP64 latency than two: whole
// calls at n = 5000, 8192 and 12000 take 372, 807 and 1580 us (int16), 547, 1299 and 2736 us
// (int32), with two 384, 893 and 1718, 620, 1357 and 2807 us; n = 3000 (int16), whose last wave is
// nearly empty then, 184 against 174 us.
template <typename WT>
__global__ void __launch_bounds__(kVerifyThreads, 3) verify_kernel(VerifyView A) {
    constexpr int VEC = 16 / sizeof(WT);
    __shared__ double tab[kExpTab];
    const VerifyParams P = *A.par;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (P.mode)
        for (int k = tid; k < kExpTab; k += kVerifyThreads) tab[k] = A.E[k];
    __syncthreads();
    const int n = A.n;
    const int j0 = (blockIdx.x * 32 + lane) * VEC;
    const int cnt = max(0, min(VEC, n - j0));
    const int r0 = (blockIdx.y * kVerifyWarps + wid) * A.rows_per_warp;
    const int r1 = min(n, r0 + A.rows_per_warp);
    double cs[VEC];
    long long vf[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) {
        cs[e] = 0.0;
        vf[e] = P.mode && e < cnt ? A.Vf[j0 + e] : 0;
    }
    for (int rb = r0; rb < r1; rb += kVerifyGroup) {
        double rs[kVerifyGroup];
        uint4 wq[kVerifyGroup];
        // the rows of the group are loaded before the first is used
#pragma unroll
        for (int r = 0; r < kVerifyGroup; ++r) {
            wq[r] = make_uint4(0u, 0u, 0u, 0u);
            if (rb + r < r1 && cnt > 0) {
                const WT* src = (const WT*)A.w + (int64_t)(rb + r) * A.ld + j0;
                if (A.vec_ok && cnt == VEC) {
                    wq[r] = __ldg((const uint4*)src);
                } else {
                    WT tmp[VEC];
#pragma unroll
                    for (int e = 0; e < VEC; ++e) tmp[e] = e < cnt ? src[e] : (WT)0;
                    unsigned* o = &wq[r].x;
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        if (sizeof(WT) == 2) o[h] = (unsigned)(unsigned short)tmp[h * VEC / 4] | ((unsigned)(unsigned short)tmp[h * VEC / 4 + 1] << 16);
                        else o[h] = (unsigned)tmp[h];
                    }
                }
            }
        }
#pragma unroll
        for (int r = 0; r < kVerifyGroup; ++r) {
            rs[r] = 0.0;
            const int row = rb + r;
            if (row >= r1) continue;
            const long long uf = P.mode ? A.Uf[row] : 0;
            const double ur = P.mode ? 0.0 : A.u[row];
            const unsigned wd[4] = {wq[r].x, wq[r].y, wq[r].z, wq[r].w};
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                const int w = sizeof(WT) == 2 ? (int)(short)(wd[e / 2] >> (16 * (e & 1))) : (int)wd[e & 3];
                double x = 0.0;
                if (w > 0) {
                    if (P.mode) x = fixed_exp2(fixed_plog<WT>(A, P, w) - uf - vf[e], P.F, tab);
                    else x = exp(A.p * log((double)w) - ur - A.v[j0 + e]);
                }
                rs[r] += x;
                cs[e] += x;
            }
        }
        // lanes 4 q .. 4 q + 3 end with the sum of row q
        const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
#pragma unroll
        for (int r = 0; r < 4; ++r) rs[r] = (b4 ? rs[r + 4] : rs[r]) + __shfl_xor_sync(0xffffffffu, b4 ? rs[r] : rs[r + 4], 16);
#pragma unroll
        for (int r = 0; r < 2; ++r) rs[r] = (b3 ? rs[r + 2] : rs[r]) + __shfl_xor_sync(0xffffffffu, b3 ? rs[r] : rs[r + 2], 8);
        double s = (b2 ? rs[1] : rs[0]) + __shfl_xor_sync(0xffffffffu, b2 ? rs[0] : rs[1], 4);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        const int row = rb + (lane >> 2);
        if ((lane & 3) == 0 && row < r1) A.rpart[(int64_t)blockIdx.x * n + row] = s;
    }
    __syncthreads();   // the table's space takes the warps' column sums
    double* cw = tab;  // [warps][32 VEC]
#pragma unroll
    for (int e = 0; e < VEC; ++e) cw[wid * 32 * VEC + lane * VEC + e] = cs[e];
    __syncthreads();
    for (int c = tid; c < 32 * VEC; c += kVerifyThreads) {
        const int j = blockIdx.x * 32 * VEC + c;
        double s = 0.0;
#pragma unroll
        for (int x = 0; x < kVerifyWarps; ++x) s += cw[x * 32 * VEC + c];
        if (j < n) A.cpart[(int64_t)blockIdx.y * n + j] = s;
    }
}

// rows (blockIdx.y = 0) or columns (1): the sum of an entry's partials and the largest
// distance from 1, not-a-number distances left out
__global__ void verify_combine_kernel(int n, int tiles, const double* rpart, int chunks, const double* cpart, double* rows,
                                      double* cols, unsigned long long* mx) {
    const int col = blockIdx.y;
    const double* part = col ? cpart : rpart;
    const int cnt = col ? chunks : tiles;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    double err = 0.0;
    if (k < n) {
        double s = 0.0;
        for (int c = 0; c < cnt; ++c) s += part[(int64_t)c * n + k];
        double* out = col ? cols : rows;
        if (out) out[k] = s;
        err = fmax(0.0, fabs(s - 1.0));
    }
    err = warp_max(err);
    // non-negative doubles order like their bit patterns
    if ((threadIdx.x & 31) == 0 && err > 0.0) atomicMax(mx + col, (unsigned long long)__double_as_longlong(err));
}

}  // namespace

sa_status verify_device(sa_ctx* ctx, const sa_matrix* a, double p, const double* d_u, const double* d_v, double* d_rows,
                        double* d_cols, double* max_row_err, double* max_col_err) {
    const int n = a->n;
    cudaStream_t st = ctx->stream;
    const bool i16 = a->wtype == SA_I16;
    const int vec = 16 / wbytes(a->wtype);
    const int tiles = (n + 32 * vec - 1) / (32 * vec);
    // rows a warp: about two waves of blocks, at most 32 rows and at least one group, but n / 128
    // for a small matrix, whose time is the chain of one lane's entries.  Whole calls at
    // n = 8, 64, 256 and 1000 (us): 59, 61, 72 and 98 (int16), 59, 61, 72 and 84 (int32);
    // 90, 95, 96 and 97, 83, 83, 88 and 87 with a group of eight rows.  With n / 256
    // n = 1000 (int32) takes 98, with n / 64 n = 512 takes 98 and 86 instead of 84 and 75.
    const int want = std::max(1, 8 * ctx->num_sms / tiles);
    int rpw = (n + want * kVerifyWarps - 1) / (want * kVerifyWarps);
    rpw = std::min(32, std::max(kVerifyGroup, (int)align_up((size_t)rpw, kVerifyGroup)));
    rpw = std::min(rpw, std::max(1, n / 128));
    const int chunks = (n + rpw * kVerifyWarps - 1) / (rpw * kVerifyWarps);
    const size_t need = 2 * align_up((size_t)n * 8, 256) + align_up((size_t)tiles * n * 8, 256) +
                        align_up((size_t)chunks * n * 8, 256) + 2 * (size_t)kVerifyTab * 8 + (size_t)kExpTab * 8 + 4096;
    sa_status rc = ctx->ws.reserve(need);
    if (rc) return rc;
    rc = ctx->pinned.reserve(64);
    if (rc) return rc;
    Carve cv(ctx->ws.ptr);
    VerifyView A{};
    long long* Uf = cv.take<long long>(n);
    long long* Vf = cv.take<long long>(n);
    long long* T = cv.take<long long>(kVerifyTab);
    double* R = cv.take<double>(kVerifyTab);
    double* E = cv.take<double>(kExpTab);
    VerifyParams* par = cv.take<VerifyParams>(1);
    unsigned long long* mx = cv.take<unsigned long long>(2);
    A.w = a->w;
    A.n = n;
    A.ld = a->ld;
    A.vec_ok = ((uintptr_t)a->w & 15) == 0 && ((size_t)a->ld * wbytes(a->wtype)) % 16 == 0;
    A.p = p;
    A.u = d_u;
    A.v = d_v;
    A.Uf = Uf;
    A.Vf = Vf;
    A.T = T;
    A.R = R;
    A.E = E;
    A.par = par;
    A.rows_per_warp = rpw;
    A.rpart = cv.take<double>((size_t)tiles * n);
    A.cpart = cv.take<double>((size_t)chunks * n);
    SA_CUDA(cudaMemsetAsync(mx, 0, 16, st));
    verify_bounds_kernel<<<1, 1024, 0, st>>>(d_u, d_v, n, p, i16 ? 15.0 : 31.0, par);
    verify_tables_kernel<<<kVerifyTab / 256, 256, 0, st>>>(d_u, d_v, n, p, par, Uf, Vf, T, R, E);
    const dim3 g(tiles, chunks);
    if (i16) verify_kernel<int16_t><<<g, kVerifyThreads, 0, st>>>(A);
    else verify_kernel<int32_t><<<g, kVerifyThreads, 0, st>>>(A);
    verify_combine_kernel<<<dim3((n + 127) / 128, 2), 128, 0, st>>>(n, tiles, A.rpart, chunks, A.cpart, d_rows, d_cols, mx);
    count_launch(4);
    SA_CUDA(cudaMemcpyAsync(ctx->pinned.ptr, mx, 16, cudaMemcpyDeviceToHost, st));
    SA_CUDA(cudaStreamSynchronize(st));
    SA_CUDA(cudaGetLastError());
    const double* h = (const double*)ctx->pinned.ptr;
    if (max_row_err) *max_row_err = h[0];
    if (max_col_err) *max_col_err = h[1];
    return SA_OK;
}

}  // namespace sa
