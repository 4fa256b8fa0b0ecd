// sweep_resident.cu -- the step kernel's iteration (sweep_step.cu) for matrices whose per-step
// matrix K fits on the chip: K stays in registers and shared memory for the sweeps of a p step.
//
// What bounds these sizes: the row pass of the streaming kernel reads K through a ring at
// 0.7 us a stage and a sweep passes two grid barriers, so a sweep took 9.0 us at n = 256,
// 11.7 us at n = 1000 and 16 us at n = 2047, of which arithmetic and L2 bytes are under 1 us.
// Here a sweep takes 3.3, 4.4 and 6 us (whole calls with their evaluations of K: 4.20 -> 1.52 ms,
// 5.40 -> 2.02 ms for 450 sweeps, 6.02 -> 2.46 ms for 360), most of it two exchanges between all blocks
// through L2 (a store and the polls that find it, about 1 us each with the blocks of both
// dies) and the chains of dependent instructions between them:
//  * block b holds its row stripe of K: the first RR rows in registers (a thread owns 4 CH columns
//    of every row, as in the streaming kernel), the others in shared memory;
//  * the row sums of all rows of the stripe are reduced together (transposed exchanges: 9
//    shuffles for eight rows), with two block barriers a sweep instead of two a stage;
//  * blocks exchange (value, sweep number) pairs in 8-byte words: a reader polls the words it
//    needs, so that the arrival of the data is the barrier and no fence, counter or second
//    trip to L2 is needed.  Column partials go to the block that owns the column; the new
//    column factors, each with a bit "within the tolerance", come back from it and decide the
//    end of the step in every block alike.
// The words of a sweep may overwrite those of the one before: a block sends its partials of
// sweep t + 1 only after it has every factor of sweep t, which their owners sent after reading
// all partials of t; and an owner sends a factor of t + 1 only after every block's partials of
// t + 1, sent after that block read its factors of t.
//
// Precision as in the streaming kernel: K in FP32 from the float-pair exponent, FP32
// multiply-adds, compensated sums of the column partials over the blocks, FP64 potentials.  The
// column total behind the next factor and the stop test is a pair of FP32 numbers (2^-47) where the
// streaming kernel forms it in FP64 and rounds factor and residual to FP32 as well; errors
// against 64 bits over the range are the streaming kernel's (3e-11 to 1e-9, both).
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "log2pair.cuh"
#include "sa_internal.h"

namespace sa {

namespace {

constexpr int kResMaxP = 64;       // p steps of a call (the schedule is a kernel parameter)
constexpr int kResMaxRows = 32;    // rows (and columns) of a block
// Copies of the column factors, each polled by its share of the blocks: with one copy the
// polls of 150 blocks queued at the few L2 lines that hold the factors and kept the owners'
// stores waiting (7000 to 9000 cycles from a store to its last reader at n = 1200 .. 2047).
constexpr int kResCopies = 16;

struct ResArgs {
    const void* w;
    int n;
    int64_t ld;
    int i16;
    float* K;                  // n x ldk staging of the register rows
    float* Lh;                 // n x ldk: log2 w as a float pair (as in the step kernel)
    float* Ll;
    int64_t ldk;
    int k0, n_p;
    float tolf;                // the largest FP32 number <= tol: the same decisions
    int max_sweeps;
    int keep_v;
    double* U;                 // in: log2 units (resumed steps), out: natural units
    double* V;
    uint64_t* part;            // [G][npad] column partials
    uint64_t* cw;              // [kResCopies][npad] column factors
    int npad;
    int smem_rows;             // rows of a stripe in shared memory at most
    unsigned* bar;             // grid barrier counter
    int* err;
    int* sweeps_out;           // n_p
    unsigned* resid_out;       // n_p, FP32 bits
    uint64_t wait_ns;
    unsigned extra_arrivals;   // testing hook, as in the step kernel
    double P[kResMaxP];
};

__device__ __forceinline__ uint64_t pack_word(float v, unsigned tag) {
    return ((uint64_t)tag << 32) | __float_as_uint(v);
}
__device__ __forceinline__ void st_word(uint64_t* p, uint64_t v) {
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint64_t ld_word(const uint64_t* p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
// two words (16-byte aligned); each word is read and written as a whole
__device__ __forceinline__ void st_word2(uint64_t* p, uint64_t a, uint64_t b) {
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void ld_word2(const uint64_t* p, uint64_t& a, uint64_t& b) {
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}

// two words of shared memory in one access; each word is read and written as a whole
__device__ __forceinline__ uint4 ld_pair(const uint4* p) {
    uint64_t a, b;
    asm volatile("ld.relaxed.cta.shared.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(smem_u32(p)) : "memory");
    return make_uint4((unsigned)a, (unsigned)(a >> 32), (unsigned)b, (unsigned)(b >> 32));
}
__device__ __forceinline__ void st_pair(uint4* p, float hi, float lo, unsigned tag) {
    asm volatile("st.relaxed.cta.shared.v2.b64 [%0], {%1, %2};" ::"r"(smem_u32(p)), "l"(pack_word(hi, tag)), "l"(pack_word(lo, tag)) : "memory");
}

// Bound of a polling loop: false once the limit is over or another block has failed.
struct PollLimit {
    uint64_t t0 = 0;
    unsigned spins = 0;
    __device__ __forceinline__ bool go_on(int* err, uint64_t wait_ns) {
        if ((++spins & 63u) != 0) return true;
        if (*(volatile int*)err != 0) return false;
        const uint64_t now = globaltimer_ns();
        if (t0 == 0) t0 = now;
        if (now - t0 > wait_ns) {
            atomicCAS(err, 0, kErrTimeout);
            return false;
        }
        return true;
    }
};

__device__ __forceinline__ unsigned float_key(float x) {
    const unsigned b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float key_float(unsigned k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// four weights of row `row` from column j (cnt of them in the matrix, zeros after)
__device__ __forceinline__ void res_load4(const ResArgs& A, int row, int j, int cnt, int w[4]) {
    const int64_t at = (int64_t)row * A.ld + j;
    if (A.i16) {
        const int16_t* p = (const int16_t*)A.w + at;
        if (cnt == 4) {
            const short4 q = *(const short4*)p;
            w[0] = q.x; w[1] = q.y; w[2] = q.z; w[3] = q.w;
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) w[e] = e < cnt ? p[e] : 0;
        }
    } else {
        const int32_t* p = (const int32_t*)A.w + at;
        if (cnt == 4) {
            const int4 q = *(const int4*)p;
            w[0] = q.x; w[1] = q.y; w[2] = q.z; w[3] = q.w;
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) w[e] = e < cnt ? p[e] : 0;
        }
    }
}

// barrier of the NT computing threads (the potentials' warp takes no part)
template <int NT>
__device__ __forceinline__ void compute_sync() {
    asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
}
template <int NT>
__device__ __forceinline__ bool compute_sync_and(bool pred) {
    unsigned r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.and.pred q, 1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((unsigned)pred), "n"(NT)
        : "memory");
    return r != 0;
}

// NT computing threads and one more warp, which keeps the FP64 potentials of the block's
// columns: a lane adds log2 S_j to V_j and hands Vs - V back as a pair of FP32 numbers for the
// next sweep's factor.  The update is some twenty dependent FP64 instructions of about a
// hundred cycles each, on the path of every sweep where the owners of the columns ran it
// themselves; on a warp of its own it passes while the next row sums are formed.
// LOADS: partial words a thread collects at most; CS: columns of a block at most (the stride
// of the collected partials: 20 keeps the eight partial sums of four columns in distinct banks).
template <int NT, int CH, int RR, int LOADS, int CS>
__global__ void __launch_bounds__(NT + 32, 1) resident_kernel(const __grid_constant__ ResArgs A) {
    constexpr int NW = NT / 32;
    constexpr int M = CH * 4;
    static_assert(RR % 2 == 0, "the rows go in pairs");
    extern __shared__ __align__(16) unsigned char res_dyn[];
    constexpr int FG = NT / 64;                   // partial sums of a column (as the streaming kernel)
    __shared__ float4 s_l2tab[256];
    __shared__ double s_ltab[256];
    __shared__ float s_red[kResMaxRows * NW];     // row partials of the warps
    __shared__ __align__(16) float s_inv[kResMaxRows];   // read four at a time
    __shared__ float s_sum[kResMaxRows];
    __shared__ double s_cref[kResMaxRows], s_u[kResMaxRows];
    __shared__ unsigned s_rmax[kResMaxRows];
    __shared__ int s_fail, s_range, s_ok;
    // between the owners and the potentials' warp, as (value, sweep number) words: the partial
    // sums of the columns and Vs - V, both as pairs; the decision (sweep number and done bit, by sweep parity)
    __shared__ uint4 s_S[CS * FG], s_D[kResMaxRows];
    __shared__ volatile unsigned s_dec[2];

    const int n = A.n, G = gridDim.x, b = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int r0 = (int)((int64_t)b * n / G), r1 = (int)((int64_t)(b + 1) * n / G);
    const int nrows = r1 - r0, c0 = r0, ncol = nrows;
    const int NC = (n + 3) / 4;
    // collection of the column partials: column fc of the block's, sources fg, fg + ng, ...
    constexpr int kShift = CS <= 8 ? 3 : 5;
    const int cw_sh = CS <= 8 || ncol <= 8 ? 3 : ncol <= 16 ? 4 : kShift;
    const int fc = tid & ((1 << cw_sh) - 1), fg = tid >> cw_sh, ng = NT >> cw_sh;
    float4* ksm = (float4*)res_dyn;                               // rows RR.. of the stripe, NC chunks each
    float* s_part = (float*)(ksm + (size_t)A.smem_rows * NC);     // [G, padded][CS]: the collected partials
    for (int j = tid; j < 256; j += NT + 32) {
        const float4 t = log2_tab_entry(j);
        s_l2tab[j] = t;
        s_ltab[j] = -log2((double)t.x);
    }
    if (tid < kResMaxRows) {
        s_inv[tid] = 0.0f;
        s_u[tid] = tid < nrows && A.k0 > 0 ? A.U[r0 + tid] : 0.0;
    }
    // partials beyond the grid stay zero
    for (int j = G * CS + tid; j < (G + 8 * FG - 1) / (8 * FG) * (8 * FG) * CS; j += NT + 32) s_part[j] = 0.0f;
    for (int j = tid; j < CS * FG; j += NT + 32) s_S[j] = make_uint4(0u, 0u, 0u, 0u);
    if (tid < kResMaxRows) s_D[tid] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) {
        s_fail = s_range = 0;
        s_dec[0] = s_dec[1] = 0u;
    }
    unsigned nbar = 1;
    if (!counter_sync(A.bar, nbar * (unsigned)G + A.extra_arrivals, A.err, &s_ok, A.wait_ns)) return;

    if (wid == NW) {
        // ---- the potentials' warp: lane l owns column c0 + l ----
        const bool own = lane < ncol;
        double v = own && A.k0 > 0 ? __ldcg(A.V + c0 + lane) : 0.0;
        unsigned t = 0;
        for (int k = A.k0; k < A.n_p; ++k) {
            const double vs = v;
            for (;;) {
                ++t;
                PollLimit lim;
                bool ok = true;
                if (own) {
                    // the FP64 sum in the streaming kernel's order
                    double S = 0.0;
#pragma unroll
                    for (int x = 0; x < FG; ++x) {
                        uint4 q = ld_pair(s_S + lane * FG + x);
                        while (ok && (q.y != t || q.w != t)) {
                            ok = lim.go_on(A.err, A.wait_ns);
                            q = ld_pair(s_S + lane * FG + x);
                        }
                        S += (double)__uint_as_float(q.x) + (double)__uint_as_float(q.z);
                    }
                    v += sum_log2(S, s_l2tab, s_ltab);
                    const double dv = vs - v;
                    const float dh = (float)dv;
                    st_pair(s_D + lane, dh, (float)(dv - (double)dh), t);
                }
                if (!__all_sync(0xffffffffu, ok)) return;
                unsigned dec;
                while (((dec = s_dec[t & 1u]) >> 1) != t)
                    if (!lim.go_on(A.err, A.wait_ns)) { ok = false; break; }
                if (!__all_sync(0xffffffffu, ok)) return;
                if (__shfl_sync(0xffffffffu, dec, 0) & 1u) break;
            }
            const bool last = k + 1 == A.n_p;
            if (own) {
                if (!last) v *= A.keep_v ? 1.0 : A.P[k + 1] / A.P[k];
                A.V[c0 + lane] = last ? v * kLn2 : v;
            }
            if (!last) {
                ++nbar;
                if (!counter_sync(A.bar, nbar * (unsigned)G + A.extra_arrivals, A.err, &s_ok, A.wait_ns)) return;
            }
        }
        return;
    }
    int cidx[CH], nval[CH];
#pragma unroll
    for (int k = 0; k < CH; ++k) {
        cidx[k] = tid + k * NT;
        nval[k] = cidx[k] < NC ? min(4, n - cidx[k] * 4) : 0;
    }
    // finalisation: threads FG c .. FG c + FG - 1 own column c0 + c
    const int col = tid / FG, grp = tid % FG;
    const bool fin_warp = wid * 32 < ncol * FG, owner = col < ncol;
    float d_own = 0.0f;   // |S - 1| of the last sweep
    // row sums: thread NW q + x adds the warps' partials of row q
    const int oc = tid / NW, ox = tid % NW;
    const uint64_t* my_cw = A.cw + (size_t)(b % kResCopies) * A.npad;

    float Kr[RR][M], cf[M];
    unsigned t = 0;   // sweeps of the launch: the tag of its words
    for (int k = A.k0; k < A.n_p; ++k) {
        const double p = A.P[k];
        const bool fresh = k == A.k0;
        // ---- evaluation of the stripe of K (see prep in sweep_step.cu) ----
        {
            // the scaled row potentials lie within cs log2 n above the row maxima: references as
            // long as the largest entry of a row stays far above the FP32 underflow, else the maxima
            double cs = k > 0 && !A.keep_v ? p / A.P[k - 1] : 0.0;
            if (cs * (double)(32 - __clz(n)) > kMaxRefShift) cs = 0.0;
            const float pf = (float)p, ph = pf, pl = (float)(p - (double)ph);
            float vh[M], vl[M];
#pragma unroll
            for (int kk = 0; kk < CH; ++kk)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const double v = e < nval[kk] && k > 0 ? __ldcg(A.V + cidx[kk] * 4 + e) : 0.0;
                    vh[4 * kk + e] = (float)v;
                    vl[4 * kk + e] = (float)(v - (double)vh[4 * kk + e]);
                }
            // log2 w of four columns of row q as float pairs (-inf: no entry)
            auto pairs = [&](int q, int kk, float lh[4], float ll[4]) {
                const int64_t at = (int64_t)(r0 + q) * A.ldk + cidx[kk] * 4;
                if (fresh) {
                    int wv[4];
                    res_load4(A, r0 + q, cidx[kk] * 4, nval[kk], wv);
                    wlog2_4(s_l2tab, wv, lh, ll);
                    *(float4*)(A.Lh + at) = make_float4(lh[0], lh[1], lh[2], lh[3]);
                    *(float4*)(A.Ll + at) = make_float4(ll[0], ll[1], ll[2], ll[3]);
                } else {
                    const float4 h = *(const float4*)(A.Lh + at), l = *(const float4*)(A.Ll + at);
                    lh[0] = h.x; lh[1] = h.y; lh[2] = h.z; lh[3] = h.w;
                    ll[0] = l.x; ll[1] = l.y; ll[2] = l.z; ll[3] = l.w;
                }
            };
            if (!(cs > 0.0)) {
                if (tid < kResMaxRows) s_rmax[tid] = float_key(-INFINITY);
                compute_sync<NT>();
                for (int q = 0; q < nrows; ++q) {
                    float m = -INFINITY;
#pragma unroll
                    for (int kk = 0; kk < CH; ++kk) {
                        if (nval[kk] == 0) continue;
                        if (fresh) {
                            int wv[4];
                            res_load4(A, r0 + q, cidx[kk] * 4, nval[kk], wv);
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (wv[e] > 0) m = fmaxf(m, fmaf(pf, lg2_approx((float)wv[e]), -vh[4 * kk + e]));
                        } else {
                            const float4 h = *(const float4*)(A.Lh + (int64_t)(r0 + q) * A.ldk + cidx[kk] * 4);
                            const float lh[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (lh[e] > -INFINITY) m = fmaxf(m, fmaf(pf, lh[e], -vh[4 * kk + e]));
                        }
                    }
                    m = warp_max(m);
                    if (lane == 0) atomicMax(&s_rmax[q], float_key(m));
                }
                compute_sync<NT>();
                if (tid < nrows) {
                    float m = key_float(s_rmax[tid]);
                    if (!(m > -INFINITY)) {
                        atomicCAS(A.err, 0, kErrNonfinite);
                        s_fail = 1;
                        m = 0.0f;
                    }
                    s_cref[tid] = (double)m;
                }
            } else if (tid < nrows) {
                s_cref[tid] = s_u[tid] * cs;
            }
            compute_sync<NT>();
            if (s_fail) return;
            for (int q = 0; q < nrows; ++q) {
                const double cref = s_cref[q];
                const float mh = (float)cref, ml = (float)(cref - (double)mh);
#pragma unroll
                for (int kk = 0; kk < CH; ++kk) {
                    if (nval[kk] == 0) continue;
                    float lh[4], ll[4], kv[4];
                    pairs(q, kk, lh, ll);
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        kv[e] = lh[e] > -INFINITY ? pair_exp2(ph, pl, make_float2(lh[e], ll[e]), vh[4 * kk + e], vl[4 * kk + e], mh, ml)
                                                  : 0.0f;
                    const float4 k4 = make_float4(kv[0], kv[1], kv[2], kv[3]);
                    if (q < RR) *(float4*)(A.K + (int64_t)(r0 + q) * A.ldk + cidx[kk] * 4) = k4;
                    else ksm[(q - RR) * NC + cidx[kk]] = k4;
                }
            }
            // the staged rows come back to the thread that wrote them
#pragma unroll
            for (int r = 0; r < RR; ++r)
#pragma unroll
                for (int kk = 0; kk < CH; ++kk) {
                    float4 k4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    if (r < nrows && nval[kk] > 0) k4 = *(const float4*)(A.K + (int64_t)(r0 + r) * A.ldk + cidx[kk] * 4);
                    Kr[r][4 * kk] = k4.x;
                    Kr[r][4 * kk + 1] = k4.y;
                    Kr[r][4 * kk + 2] = k4.z;
                    Kr[r][4 * kk + 3] = k4.w;
                }
#pragma unroll
            for (int m = 0; m < M; ++m) cf[m] = (m % 4) < nval[m / 4] ? 1.0f : 0.0f;
            compute_sync<NT>();   // threads beyond the row read its last chunk (times a zero factor)
        }
        // ---- sweeps ----
        int sweeps = 0;
        bool done = false;
        while (!done) {
            ++t;
            // row sums s_q = sum_j K_qj c_j of the stripe, eight rows at a time
            auto dot = [&](const float4& kv, int kk, float& a0, float& a1) {
                a0 = fmaf(kv.x, cf[4 * kk], a0);
                a1 = fmaf(kv.y, cf[4 * kk + 1], a1);
                a0 = fmaf(kv.z, cf[4 * kk + 2], a0);
                a1 = fmaf(kv.w, cf[4 * kk + 3], a1);
            };
            // the sums of rows q0 .. q0 + 7 below `end`: a row's word is stored by the group that owns
            // it alone (RR need not be a multiple of eight, and two lanes' stores to one word
            // are not ordered)
            auto reduce8 = [&](float s[8], int q0, int end) {
                const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
#pragma unroll
                for (int r = 0; r < 4; ++r) s[r] = (b4 ? s[r + 4] : s[r]) + __shfl_xor_sync(0xffffffffu, b4 ? s[r] : s[r + 4], 16);
#pragma unroll
                for (int r = 0; r < 2; ++r) s[r] = (b3 ? s[r + 2] : s[r]) + __shfl_xor_sync(0xffffffffu, b3 ? s[r] : s[r + 2], 8);
                float x = (b2 ? s[1] : s[0]) + __shfl_xor_sync(0xffffffffu, b2 ? s[0] : s[1], 4);
                x += __shfl_xor_sync(0xffffffffu, x, 2);
                x += __shfl_xor_sync(0xffffffffu, x, 1);
                const int q = q0 + (lane >> 2);
                if ((lane & 3) == 0 && q < end) s_red[q * NW + wid] = x;
            };
#pragma unroll
            for (int g = 0; g < (RR + 7) / 8; ++g) {
                if (8 * g >= min(nrows, RR)) break;
                float s[8];
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    float a0 = 0.0f, a1 = 0.0f;
                    if (8 * g + r < RR) {
                        const float* kr = Kr[min(8 * g + r, RR - 1)];
#pragma unroll
                        for (int kk = 0; kk < CH; ++kk)
                            dot(make_float4(kr[4 * kk], kr[4 * kk + 1], kr[4 * kk + 2], kr[4 * kk + 3]), kk, a0, a1);
                    }
                    s[r] = a0 + a1;
                }
                reduce8(s, 8 * g, RR);
            }
            for (int q0 = RR; q0 < nrows; q0 += 8) {
                float s[8];
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    float a0 = 0.0f, a1 = 0.0f;
#pragma unroll
                    for (int kk = 0; kk < CH; ++kk)
                        // beyond the row c is zero, beyond the stripe the sum is not used
                        dot(ksm[(min(q0 + r, nrows - 1) - RR) * NC + min(cidx[kk], NC - 1)], kk, a0, a1);
                    s[r] = a0 + a1;
                }
                reduce8(s, q0, nrows);
            }
            compute_sync<NT>();
            {
                float s = 0.0f;
                if (oc < nrows && ox < 4) {
#pragma unroll
                    for (int x = 0; x < NW; x += 4) s += s_red[oc * NW + ox + x];
                }
                s += __shfl_xor_sync(0xffffffffu, s, 1);
                s += __shfl_xor_sync(0xffffffffu, s, 2);
                if (ox == 0 && oc < nrows) {
                    if (!(s >= 0x1p-120f && s <= 0x1p120f)) {
                        atomicCAS(A.err, 0, kErrNonfinite);
                        s_range = 1;
                    }
                    s_sum[oc] = s;
                    s_inv[oc] = rcp_approx(s);
                }
            }
            compute_sync<NT>();
            // a flag that only the lines above set: s_fail may already be set by a thread in the polls
            // below while another has not read it here, and the threads that stay would wait
            // for the one that left
            if (s_range) return;
            // column partials c_j sum_q K_qj / s_q, the rows in the streaming kernel's order (pairs
            // of rows, last pair first in the first sweep of a step and in every other one after), so
            // that the kernels' FP32 sums round alike
            float S[M];
#pragma unroll
            for (int m = 0; m < M; ++m) S[m] = 0.0f;
            auto add_smem = [&](int q) {   // rows q, q + 1 (the second may lie beyond the stripe)
                const float inv0 = s_inv[q], inv1 = q + 1 < nrows ? s_inv[q + 1] : 0.0f;
                const float4* k0 = ksm + (q - RR) * NC;
                const float4* k1 = ksm + (min(q + 1, nrows - 1) - RR) * NC;
                float4 a[CH], c[CH];
#pragma unroll
                for (int kk = 0; kk < CH; ++kk) {
                    a[kk] = k0[min(cidx[kk], NC - 1)];
                    c[kk] = k1[min(cidx[kk], NC - 1)];
                }
#pragma unroll
                for (int kk = 0; kk < CH; ++kk) {
                    S[4 * kk] = fmaf(c[kk].x, inv1, fmaf(a[kk].x, inv0, S[4 * kk]));
                    S[4 * kk + 1] = fmaf(c[kk].y, inv1, fmaf(a[kk].y, inv0, S[4 * kk + 1]));
                    S[4 * kk + 2] = fmaf(c[kk].z, inv1, fmaf(a[kk].z, inv0, S[4 * kk + 2]));
                    S[4 * kk + 3] = fmaf(c[kk].w, inv1, fmaf(a[kk].w, inv0, S[4 * kk + 3]));
                }
            };
            if (sweeps & 1) {
#pragma unroll
                for (int g = 0; g < (RR + 3) / 4; ++g) {
                    const float4 i4 = *(const float4*)(s_inv + 4 * g);   // zero beyond the stripe
                    const float inv[4] = {i4.x, i4.y, i4.z, i4.w};
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int m = 0; m < M; ++m)
                            if (4 * g + r < RR) S[m] = fmaf(Kr[min(4 * g + r, RR - 1)][m], inv[r], S[m]);
                }
                for (int q = RR; q < nrows; q += 2) add_smem(q);
            } else {
                for (int q = (nrows - 1) & ~1; q >= RR; q -= 2) add_smem(q);
#pragma unroll
                for (int g = (RR + 3) / 4 - 1; g >= 0; --g) {
                    const float4 i4 = *(const float4*)(s_inv + 4 * g);   // zero beyond the stripe
                    const float inv[4] = {i4.x, i4.y, i4.z, i4.w};
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        constexpr int kBack[4] = {2, 3, 0, 1};
                        const int x = kBack[r];
#pragma unroll
                        for (int m = 0; m < M; ++m)
                            if (4 * g + x < RR) S[m] = fmaf(Kr[min(4 * g + x, RR - 1)][m], inv[x], S[m]);
                    }
                }
            }
#pragma unroll
            for (int kk = 0; kk < CH; ++kk)
                if (nval[kk] > 0) {
                    uint64_t* o = A.part + (size_t)b * A.npad + cidx[kk] * 4;
                    st_word2(o, pack_word(S[4 * kk] * cf[4 * kk], t), pack_word(S[4 * kk + 1] * cf[4 * kk + 1], t));
                    st_word2(o + 2, pack_word(S[4 * kk + 2] * cf[4 * kk + 2], t), pack_word(S[4 * kk + 3] * cf[4 * kk + 3], t));
                }
            // ---- the block's own columns: every block's partials as they arrive ----
            {
                const uint64_t* src = A.part + c0 + fc;
                uint64_t w[LOADS];
                const int cnt = fc < ncol ? (G - fg + ng - 1) / ng : 0;   // words this thread collects
#pragma unroll
                for (int l = 0; l < LOADS; ++l)
                    w[l] = l < cnt ? ld_word(src + (size_t)(fg + l * ng) * A.npad) : (uint64_t)t << 32;
                PollLimit lim;
                for (;;) {
                    bool miss = false;
#pragma unroll
                    for (int l = 0; l < LOADS; ++l)
                        if ((unsigned)(w[l] >> 32) != t) {
                            w[l] = ld_word(src + (size_t)(fg + l * ng) * A.npad);
                            miss = true;
                        }
                    if (!miss) break;
                    if (!lim.go_on(A.err, A.wait_ns)) { s_fail = 1; break; }
                }
                if (fc < ncol) {
#pragma unroll
                    for (int l = 0; l < LOADS; ++l)
                        if (l < cnt) s_part[(fg + l * ng) * CS + fc] = __uint_as_float((unsigned)w[l]);
                }
                compute_sync<NT>();
                if (fin_warp) {
                    // the streaming kernel's order: sources grp, grp + FG, ... compensated
                    float s = 0.0f, c = 0.0f;
                    if (owner) {
                        // (a zero changes neither s - c nor its compensation); eight loads ahead
                        // of the chain of dependent additions
                        const float* ps = s_part + grp * CS + col;
                        for (int g0 = 0; g0 < G; g0 += 8 * FG, ps += 8 * FG * CS) {
                            float a[8];
#pragma unroll
                            for (int x = 0; x < 8; ++x) a[x] = ps[x * FG * CS];
#pragma unroll
                            for (int x = 0; x < 8; ++x) {
                                const float y = a[x] - c;
                                const float z = s + y;
                                c = (z - s) - y;
                                s = z;
                            }
                        }
                    }
                    float hi = s, lo = -c;
                    const float raw_hi = hi, raw_lo = lo;
#pragma unroll
                    for (int o = 1; o < FG; o <<= 1)
                        pair_add(hi, lo, __shfl_xor_sync(0xffffffffu, hi, o), __shfl_xor_sync(0xffffffffu, lo, o));
                    if (owner) {
                        float e;
                        hi = two_sum(hi, lo, &e);
                        lo = e;
                        unsigned tag = t << 2;
                        d_own = fabsf((hi - 1.0f) + lo);
                        if (d_own <= A.tolf) tag |= 1u;
                        // c = 2^(Vs - V - log2 S), the exponent as a pair of FP32 numbers
                        float dh = 0.0f, dl = 0.0f;
                        if (sweeps > 0) {
                            uint4 q = ld_pair(s_D + col);
                            PollLimit lim;
                            while (q.y != t - 1u || q.w != t - 1u) {
                                if (!lim.go_on(A.err, A.wait_ns)) { s_fail = 1; break; }
                                q = ld_pair(s_D + col);
                            }
                            dh = __uint_as_float(q.x);
                            dl = __uint_as_float(q.z);
                        }
                        // the potentials' warp is done with the last sweep's sums once Vs - V is there
                        st_pair(s_S + col * FG + grp, raw_hi, raw_lo, t);
                        const float2 lg = pair_log2(hi, lo, s_l2tab);
                        const float x = two_sum(dh, -lg.x, &e);
                        float c_new = ex2_approx(x + (e + (dl - lg.y)));
                        if (!(hi >= 0x1p-126f) || !(hi < INFINITY)) {
                            if (!(hi > 0.0f) || !(hi < INFINITY)) {
                                atomicCAS(A.err, 0, kErrNonfinite);
                                tag |= 2u;
                            } else {
                                // a sum below the normal numbers, where pair_log2 finds no exponent: scaled, and
                                // to the FP32 rounding of an exponent near 127; a factor beyond 2^127 is cut (the
                                // potentials do not use it: the next sweep makes up for it)
                                c_new = ex2_approx(fminf(dh + (dl + (64.0f - lg2_approx(hi * 0x1p64f))), 127.0f));
                            }
                        }
                        const uint64_t word = pack_word(c_new, tag);
                        for (int r = grp; r < kResCopies; r += FG) st_word(A.cw + (size_t)r * A.npad + c0 + col, word);
                    }
                }
            }
            // the other warps wait here, not in polls that would take the owners' issue slots: no
            // factor is due before the block's own are out
            compute_sync<NT>();
            // ---- the new column factors as they arrive ----
            bool within = true, bad = false;
            {
                uint64_t w[M];
#pragma unroll
                for (int m = 0; m < M; ++m) w[m] = (m % 4) < nval[m / 4] ? 0ull : (uint64_t)((t << 2) | 1u) << 32;
                PollLimit lim;
                for (;;) {
                    bool miss = false;
#pragma unroll
                    for (int kk = 0; kk < CH; ++kk)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint64_t& w0 = w[4 * kk + 2 * h];
                            uint64_t& w1 = w[4 * kk + 2 * h + 1];
                            if ((unsigned)(w0 >> 34) != t || (unsigned)(w1 >> 34) != t) {
                                uint64_t x0, x1;
                                ld_word2(my_cw + cidx[kk] * 4 + 2 * h, x0, x1);
                                w0 = x0;
                                if (2 * h + 1 < nval[kk]) w1 = x1;
                                miss |= (unsigned)(w0 >> 34) != t || (unsigned)(w1 >> 34) != t;
                            }
                        }
                    if (!miss) break;
                    if (!lim.go_on(A.err, A.wait_ns)) { s_fail = 1; break; }
                }
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    const bool real = (m % 4) < nval[m / 4];
                    cf[m] = real ? __uint_as_float((unsigned)w[m]) : 0.0f;
                    within = within && ((w[m] >> 32) & 1u);
                    bad = bad || ((w[m] >> 33) & 1u);
                }
                if (bad) s_fail = 1;   // its owner has recorded the error
            }
            ++sweeps;
            const bool all = compute_sync_and<NT>(within);
            if (s_fail) return;
            done = all || sweeps >= A.max_sweeps;
            if (tid == 0) s_dec[t & 1u] = (t << 1) | (done ? 1u : 0u);
        }
        // ---- end of the step ----
        const bool last = k + 1 == A.n_p;
        if (tid < nrows) {
            const double u = s_cref[tid] + log2((double)s_sum[tid]);   // as the streaming kernel, to the last bit
            s_u[tid] = u;
            if (last) A.U[r0 + tid] = u * kLn2;
        }
        if (owner && grp == 0) atomicMax(A.resid_out + k, __float_as_uint(d_own));   // non-negative floats order like their bits
        if (b == 0 && tid == 0) A.sweeps_out[k] = sweeps;
        if (!last) {
            ++nbar;
            if (!counter_sync(A.bar, nbar * (unsigned)G + A.extra_arrivals, A.err, &s_ok, A.wait_ns)) return;
        }
    }
}

struct ResCfg {
    int nt = 0, ch = 0, rr = 0, loads = 0, cs = 0, grid = 0, smem_rows = 0;
    size_t smem = 0;
};

// static shared memory of the kernels, rounded up (the tables and reductions)
constexpr size_t kResStatic = 14 * 1024;

ResCfg pick_resident(const sa_ctx* ctx, int n) {
    ResCfg c;
    const int nc = (n + 3) / 4;
    int G = std::max(1, std::min(ctx->num_sms, n / 8));
    if (ctx->max_grid > 0) G = std::min(G, ctx->max_grid);
    const int rows = (n + G - 1) / G;
    if (nc <= 128) c = {128, 1, 16, 8, rows <= 8 ? 8 : 20};
    else if (nc <= 256) c = {256, 1, 16, 8, rows <= 8 ? 8 : 20};
    else if (nc <= 512 && rows <= 8) c = {512, 1, 8, 5, 8};
    else if (nc <= 512) c = {512, 1, 14, 5, 20};
    else if (nc <= 1024) c = {512, 2, 8, 10, 32};
    else return c;
    c.grid = G;
    const int cw = rows <= 8 ? 8 : rows <= 16 ? 16 : 32, pad = c.nt / 8;
    c.smem_rows = std::max(0, rows - c.rr);
    c.smem = (size_t)c.smem_rows * nc * 16 + (size_t)(G + pad - 1) / pad * pad * c.cs * 4;
    const bool ok = rows <= c.cs && c.smem + kResStatic <= ctx->smem_optin &&
                    (G + c.nt / cw - 1) / (c.nt / cw) <= c.loads;
    if (!ok) c.nt = 0;
    return c;
}

template <int NT, int CH, int RR, int LOADS, int CS>
sa_status launch_resident(sa_ctx* ctx, const ResArgs& args, const ResCfg& cfg) {
    auto kern = resident_kernel<NT, CH, RR, LOADS, CS>;
    SA_CUDA(allow_dynamic_smem(kern, ctx->smem_optin));
    void* params[] = {(void*)&args};
    SA_CUDA(cudaLaunchCooperativeKernel((const void*)kern, dim3(cfg.grid), dim3(NT + 32), params, cfg.smem, ctx->stream));
    count_launch();
    return SA_OK;
}

}  // namespace

// The resident kernel takes a call of scale_step that needs no sparse epochs, whose schedule fits
// its parameters, whose sweeps fit the words' tags (30 bits) and whose stripes fit the SMs (n up to about 3400 on a full GB300; fewer
// with a capped grid).
bool resident_supported(const sa_ctx* ctx, const sa_matrix* a, const sa_scale_opts* o) {
    return !ctx->step_sparse && o->n_p <= kResMaxP && (int64_t)o->n_p * o->max_sweeps_per_p < (1ll << 30) &&
           pick_resident(ctx, a->n).nt > 0;
}

sa_status scale_resident(sa_ctx* ctx, const sa_matrix* a, const sa_scale_opts* o, double* U, double* V, sa_scale_info* info) {
    const int n = a->n;
    const ResCfg cfg = pick_resident(ctx, n);
    cudaStream_t st = ctx->stream;
    const int npad = (int)align_up((size_t)n, 32);
    const int64_t ldk = (int64_t)align_up((size_t)n, 4);
    const size_t plane = align_up((size_t)n * ldk * 4, 256);
    const size_t part_bytes = align_up((size_t)cfg.grid * npad * 8, 256), cw_bytes = align_up((size_t)kResCopies * npad * 8, 256);
    const size_t ctl_bytes = 1024;   // barrier, error, sweeps and residuals of up to 64 steps
    sa_status rc = ctx->ws.reserve(3 * plane + part_bytes + cw_bytes + ctl_bytes + 4096);
    if (rc) return rc;
    rc = ctx->pinned.reserve(ctl_bytes);
    if (rc) return rc;
    Carve cv(ctx->ws.ptr);
    // words and control block are contiguous: one clear
    ResArgs args{};
    args.part = cv.take<uint64_t>(part_bytes / 8);
    args.cw = cv.take<uint64_t>(cw_bytes / 8);
    unsigned* ctl = cv.take<unsigned>(ctl_bytes / 4);
    args.bar = ctl;
    args.err = (int*)(ctl + 32);
    args.sweeps_out = (int*)(ctl + 64);
    args.resid_out = ctl + 128;
    args.K = cv.take<float>(plane / 4);
    args.Lh = cv.take<float>(plane / 4);
    args.Ll = cv.take<float>(plane / 4);
    args.w = a->w;
    args.n = n;
    args.ld = a->ld;
    args.i16 = a->wtype == SA_I16;
    args.ldk = ldk;
    args.k0 = o->resume_from > 0 ? o->resume_from : 0;
    args.n_p = o->n_p;
    args.tolf = (float)o->tol;
    if ((double)args.tolf > o->tol) args.tolf = std::nextafter(args.tolf, 0.0f);
    args.max_sweeps = o->max_sweeps_per_p;
    args.keep_v = o->warm_keep_v;
    args.U = U;
    args.V = V;
    args.npad = npad;
    args.smem_rows = cfg.smem_rows;
    args.wait_ns = ctx->wait_ns;
    args.extra_arrivals = ctx->test_unreachable_barrier ? 1u : 0u;
    std::copy(o->p, o->p + o->n_p, args.P);
    const int k0 = args.k0;
    SA_CUDA(cudaMemsetAsync(args.part, 0, (char*)(ctl + ctl_bytes / 4) - (char*)args.part, st));
    if (k0 > 0 && !o->warm_keep_v) launch_scale_vec(V, n, o->p[k0] / o->p[k0 - 1], st);
    cudaEvent_t ev0, ev1;
    SA_CUDA(cudaEventCreate(&ev0));
    SA_CUDA(cudaEventCreate(&ev1));
    SA_CUDA(cudaEventRecord(ev0, st));
    if (cfg.nt == 128 && cfg.cs == 8) rc = launch_resident<128, 1, 16, 8, 8>(ctx, args, cfg);
    else if (cfg.nt == 128) rc = launch_resident<128, 1, 16, 8, 20>(ctx, args, cfg);
    else if (cfg.nt == 256 && cfg.cs == 8) rc = launch_resident<256, 1, 16, 8, 8>(ctx, args, cfg);
    else if (cfg.nt == 256) rc = launch_resident<256, 1, 16, 8, 20>(ctx, args, cfg);
    else if (cfg.cs == 8) rc = launch_resident<512, 1, 8, 5, 8>(ctx, args, cfg);
    else if (cfg.ch == 1) rc = launch_resident<512, 1, 14, 5, 20>(ctx, args, cfg);
    else rc = launch_resident<512, 2, 8, 10, 32>(ctx, args, cfg);
    if (rc) { cudaEventDestroy(ev0); cudaEventDestroy(ev1); return rc; }
    SA_CUDA(cudaEventRecord(ev1, st));
    unsigned* h = (unsigned*)ctx->pinned.ptr;
    SA_CUDA(cudaMemcpyAsync(h, ctl, ctl_bytes, cudaMemcpyDeviceToHost, st));
    SA_CUDA(cudaStreamSynchronize(st));
    float kms = 0.0f;
    SA_CUDA(cudaEventElapsedTime(&kms, ev0, ev1));
    cudaEventDestroy(ev0);
    cudaEventDestroy(ev1);
    const int err = (int)h[32];
    const float* resid = (const float*)(h + 128);
    int64_t total = 0;
    int conv = 1;
    for (int k = k0; k < o->n_p; ++k) {
        total += (int)h[64 + k];
        if (!((double)resid[k] <= o->tol)) conv = 0;
    }
    if (info) {
        info->sweeps_total = total;
        info->residual = resid[o->n_p - 1];
        info->p_final = o->p[o->n_p - 1];
        info->converged = conv;
        info->steps_done = o->n_p - k0;
        info->kernel_used = SA_KERNEL_STEP;
        info->kernel_ms = kms;
    }
    if (err == kErrTimeout) {
        set_error("step sweep: a bounded device wait timed out (grid of %d blocks)", cfg.grid);
        return SA_E_TIMEOUT;
    }
    if (err == kErrNonfinite) {
        set_error("step sweep: a row or column sum left the FP32 range (matrix without support?)");
        return SA_E_NONFINITE;
    }
    return conv ? SA_OK : SA_E_NOT_CONVERGED;
}

}  // namespace sa
