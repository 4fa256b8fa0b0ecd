// batch_cluster.cuh -- one instance of the batched form (n <= 512) on one block, or on a cluster
// of two or four, that holds its per-step matrix K on the chip (Sec. 4.1.2 iteration in log
// coordinates, Sec. 4.2 stop rule, the deformed warm start of Sec. 4.1 between p steps).
//
// What bounds these sizes: with K in a global slot per block (two blocks per SM, 0.57 MB of K an
// instance between n = 257 and 512) the slots in flight exceeded the L2, and a sweep was one
// read of K at 4.6 TB/s: 26 ms for the larger bucket of the 4096-instance workload, 6 ms for the one
// below.  Here RG rows a warp stay in registers and RS in shared memory.  n <= 144 takes half an SM
// (eight warps), n <= 256 two halves, n <= 384 two SMs and n <= 512 four (sixteen warps each): a sweep
// takes 3.3, 2.5, 3.2 and 3.6 us with every SM busy, its arithmetic 0.5 us of that, the rest
// the chains of its reductions and the exchange between the blocks.  Measured and dropped:
// clusters of four and eight half SMs for the larger sizes (5.0 and 5.3 us), and one block per
// SM that streams what does not fit from L2 (10 us at n = 380, 25 us at n = 510 for 152 instances:
// 5 to 7.6 TB/s).
//
// Block r of the cluster owns the rows [r n/C, (r+1) n/C); warp w of a block the rows w, w + NW,
// ... of these, lane l the 16-byte column chunks l, l + 32, ... of every row.  Row sums of eight
// rows are reduced together; the column partials of the warps meet in shared memory (two
// rounds of half the warps), a thread per chunk of four columns adds them and
// sends its block's sums to every block of the cluster, and after the cluster barrier each
// block forms the same totals, factors and decisions.  The column potentials stay in FP64: each
// block updates its share at the end of a p step.  log2 w is formed once per instance as a
// float pair and kept in the slot (8 bytes per entry, read once per p step).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "log2pair.cuh"
#include "sa_internal.h"

namespace sa {

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// all threads of the cluster; their shared-memory writes before it, local and remote, are
// visible after it
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// shared address of the same variable in block `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_map(const void* p, unsigned rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void cluster_st4(uint32_t addr, float4 v) {   // 16-byte aligned
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void cluster_st(uint32_t addr, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_st(uint32_t addr, int v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// CH: 16-byte column chunks a lane (n <= 128 CH); RG: rows a warp in registers; RS: rows a
// warp in shared memory at most (NW C (RG + RS) >= the largest n).
template <int NT, int C, int CH, int RG, int RS>
struct __align__(16) ClusterSmem {
    static constexpr int NW = NT / 32;
    static constexpr int NMAX = 128 * CH;
    float4 l2tab[256];
    double ltab[256];
    double V[(NMAX + C - 1) / C + 1];       // this block's share of the column potentials
    // 16-byte aligned: read and written as float4
    __align__(16) float K[RS * NW][NMAX];           // rows RG + s of warp w at [s 8 + w]
    __align__(16) float colpart[NW / 2][NMAX];
    __align__(16) float inbox[2][C > 1 ? C - 1 : 1][C > 1 ? NMAX : 4];   // the other blocks' column sums, by sweep parity
    __align__(16) float c[NMAX];
    float srow[(NMAX + C - 1) / C], Cr[(NMAX + C - 1) / C];   // the block's row sums and references
    int inst, bad, badk;
    // V as float pairs during an evaluation of K, in the (then idle) partial sums
    __device__ __forceinline__ float* vhi() { return colpart[0]; }
    __device__ __forceinline__ float* vlo() { return colpart[1]; }
};

// Scales instance after instance of the queue: the arguments are those of the batched kernels
// (batch.cu); slot: this cluster's global slot of 3 n ceil(n/4)*4 floats.
template <typename WT, int NT, int C, int CH, int RG, int RS, typename Args>
__device__ __forceinline__ void cluster_instances(const Args& A, float* slot) {
    using Smem = ClusterSmem<NT, C, CH, RG, RS>;
    constexpr int NW = NT / 32, NMAX = Smem::NMAX, M = 4 * CH;
    constexpr int RW = RG + RS;
    // finalisation: thread t of the first 32 CH, and its twins at a distance of TW, hold the four
    // columns of chunk t; a twin sends their sums to its share of the blocks
    constexpr int TW = CH <= 2 ? 64 : 128, TWINS = NT / TW;
    extern __shared__ __align__(16) unsigned char cl_dyn[];
    Smem& sm = *(Smem*)cl_dyn;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned rank = C > 1 ? cluster_rank() : 0u;
    const int chunk = tid & (TW - 1), twin = tid / TW;
    for (int j = tid; j < 256; j += NT) {
        const float4 t = log2_tab_entry(j);
        sm.l2tab[j] = t;
        sm.ltab[j] = -log2((double)t.x);
    }
    auto sync_all = [&]() {
        if (C > 1) cluster_sync();
        else __syncthreads();
    };
    sync_all();   // the cluster's blocks run (their shared memory may be written)
    for (;;) {
        if (rank == 0 && tid == 0) {
            const unsigned q = atomicAdd(A.queue, 1u);
            const int inst = q < (unsigned)A.k ? A.order[q] : -1;
            sm.inst = inst;
#pragma unroll
            for (int r = 1; r < C; ++r) cluster_st(cluster_map(&sm.inst, r), inst);
        }
        if (tid == 0) sm.bad = sm.badk = 0;
        sync_all();
        const int inst = sm.inst;
        if (inst < 0) return;
        const int n = A.n[inst];
        const int64_t ld = A.ld[inst];
        const WT* wb = (const WT*)A.w[inst];
        const int NC = (n + 3) / 4, ldk = NC * 4;
        const int r0 = (int)rank * n / C, r1 = ((int)rank + 1) * n / C, nrows = r1 - r0;
        // columns whose potentials this block keeps
        const int v0 = (int)rank * n / C, v1 = ((int)rank + 1) * n / C;
        float* Kg = slot;                           // staging of the register rows
        float* Lh = slot + (size_t)n * ldk;         // log2 w as a float pair
        float* Ll = Lh + (size_t)n * ldk;
        for (int j = v0 + tid; j < v1; j += NT) sm.V[j - v0] = 0.0;
        for (int j = tid; j < NMAX; j += NT) {
            sm.vhi()[j] = sm.vlo()[j] = 0.0f;
        }
        __syncthreads();
        // log2 w of the block's rows: a loop of its own, since it runs once
        for (int q = wid; q < nrows; q += NW)
#pragma unroll 1
            for (int c4 = lane; c4 < NC; c4 += 32) {
                const WT* wr = wb + (int64_t)(r0 + q) * ld + 4 * c4;
                int w[4];
                float lh[4], ll[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) w[e] = 4 * c4 + e < n ? (int)wr[e] : 0;
                wlog2_4(sm.l2tab, w, lh, ll);
                *(float4*)(Lh + (int64_t)(r0 + q) * ldk + 4 * c4) = make_float4(lh[0], lh[1], lh[2], lh[3]);
                *(float4*)(Ll + (int64_t)(r0 + q) * ldk + 4 * c4) = make_float4(ll[0], ll[1], ll[2], ll[3]);
            }
        float Kr[RG][M];
        int sweeps_all = 0;
        bool bad = false, capped = false;
        for (int k = 0; k < A.n_p && !bad; ++k) {
            const double p = A.P[k];
            // ---- evaluation of the block's rows of K: one rolled loop (unrolled for the register rows it
            //      was bound by instruction fetches), the next row's pairs prefetched ----
            const float ph = (float)p, pl = (float)(p - (double)ph);
#pragma unroll 1
            for (int r = 0; r < RW; ++r) {
                const int q = wid + NW * r;
                const bool live = q < nrows;
                const int64_t row = r0 + q;
                if (q + NW < nrows) {
#pragma unroll
                    for (int kk = 0; kk < CH; ++kk)
                        if (lane + 32 * kk < NC) {
                            const int64_t at = (row + NW) * ldk + 4 * (lane + 32 * kk);
                            asm volatile("prefetch.global.L1 [%0];" ::"l"(Lh + at));
                            asm volatile("prefetch.global.L1 [%0];" ::"l"(Ll + at));
                        }
                }
                float4 lh[CH], ll[CH];
                float m = -INFINITY;
#pragma unroll
                for (int kk = 0; kk < CH; ++kk) {
                    const int c4 = lane + 32 * kk;
                    lh[kk] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
                    ll[kk] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    if (live && c4 < NC) {
                        lh[kk] = *(const float4*)(Lh + row * ldk + 4 * c4);
                        ll[kk] = *(const float4*)(Ll + row * ldk + 4 * c4);
                    }
                }
#pragma unroll
                for (int kk = 0; kk < CH; ++kk) {
                    const float4 vh = *(const float4*)(sm.vhi() + 4 * (lane + 32 * kk));
                    // an absent entry's -inf stays -inf
                    m = fmaxf(fmaxf(m, fmaxf(fmaf(ph, lh[kk].x, -vh.x), fmaf(ph, lh[kk].y, -vh.y))),
                              fmaxf(fmaf(ph, lh[kk].z, -vh.z), fmaf(ph, lh[kk].w, -vh.w)));
                }
                m = warp_max(m);
                if (!(m > -INFINITY)) {
                    if (live) sm.badk = 1;
                    m = 0.0f;
                }
                if (live && lane == 0) sm.Cr[q] = m;
#pragma unroll
                for (int kk = 0; kk < CH; ++kk) {
                    const int c4 = lane + 32 * kk;
                    const float4 vh = *(const float4*)(sm.vhi() + 4 * c4), vl = *(const float4*)(sm.vlo() + 4 * c4);
                    auto one = [&](float h, float l, float a, float b) {
                        return h > -INFINITY ? pair_exp2(ph, pl, make_float2(h, l), a, b, m, 0.0f) : 0.0f;
                    };
                    const float4 k4 = make_float4(one(lh[kk].x, ll[kk].x, vh.x, vl.x), one(lh[kk].y, ll[kk].y, vh.y, vl.y),
                                                  one(lh[kk].z, ll[kk].z, vh.z, vl.z), one(lh[kk].w, ll[kk].w, vh.w, vl.w));
                    if (r >= RG) *(float4*)&sm.K[(r - RG) * NW + wid][4 * c4] = k4;   // zeros past the stripe
                    else if (live && c4 < NC) *(float4*)(Kg + row * ldk + 4 * c4) = k4;
                }
            }
#pragma unroll
            for (int r = 0; r < RG; ++r) {
                const int q = wid + NW * r;
#pragma unroll
                for (int kk = 0; kk < CH; ++kk) {
                    const int c4 = lane + 32 * kk;
                    float4 k4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    if (q < nrows && c4 < NC) k4 = *(const float4*)(Kg + (int64_t)(r0 + q) * ldk + 4 * c4);
                    Kr[r][4 * kk] = k4.x; Kr[r][4 * kk + 1] = k4.y; Kr[r][4 * kk + 2] = k4.z; Kr[r][4 * kk + 3] = k4.w;
                }
            }
            float cj[4];   // the factors of the thread's chunk
#pragma unroll
            for (int e = 0; e < 4; ++e) cj[e] = 4 * chunk + e < n ? 1.0f : 0.0f;
            for (int j = tid; j < NMAX; j += NT) sm.c[j] = j < n ? 1.0f : 0.0f;
            __syncthreads();
            // ---- sweeps ----
            int sweeps = 0;
            bool done = false;
            while (!done) {
                const int par = sweeps & 1;
                float cf[M], S[M];
#pragma unroll
                for (int kk = 0; kk < CH; ++kk) {
                    const float4 c4 = *(const float4*)(sm.c + 4 * (lane + 32 * kk));
                    cf[4 * kk] = c4.x; cf[4 * kk + 1] = c4.y; cf[4 * kk + 2] = c4.z; cf[4 * kk + 3] = c4.w;
                }
#pragma unroll
                for (int x = 0; x < M; ++x) S[x] = 0.0f;
                int badr = sm.badk;
                auto dot4 = [&](const float4& q, int kk, float a[2]) {
                    a[0] = fmaf(q.x, cf[4 * kk], a[0]);
                    a[1] = fmaf(q.y, cf[4 * kk + 1], a[1]);
                    a[0] = fmaf(q.z, cf[4 * kk + 2], a[0]);
                    a[1] = fmaf(q.w, cf[4 * kk + 3], a[1]);
                };
                // eight rows of the warp at a time: their sums are reduced together (each exchange
                // halves the rows a lane carries: nine shuffles, not forty), the reciprocals come
                // back by eight independent shuffles, and rows in shared memory are read again
#pragma unroll
                for (int g = 0; g < RW; g += 8) {
                    if (wid + NW * g >= nrows) break;
                    float d[8];
#pragma unroll
                    for (int r = 0; r < 8; ++r) {
                        float a[2] = {0.0f, 0.0f};
                        if (g + r < RG) {
                            const float* kr = Kr[g + r < RG ? g + r : 0];
#pragma unroll
                            for (int kk = 0; kk < CH; ++kk)
                                dot4(make_float4(kr[4 * kk], kr[4 * kk + 1], kr[4 * kk + 2], kr[4 * kk + 3]), kk, a);
                        } else if (g + r < RW) {   // rows beyond the block's hold zeros
                            const float* kr = sm.K[(g + r - RG) * NW + wid];
#pragma unroll
                            for (int kk = 0; kk < CH; ++kk) dot4(*(const float4*)(kr + 4 * (lane + 32 * kk)), kk, a);
                        }
                        d[r] = a[0] + a[1];
                    }
                    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
#pragma unroll
                    for (int r = 0; r < 4; ++r) d[r] = (b4 ? d[r + 4] : d[r]) + __shfl_xor_sync(0xffffffffu, b4 ? d[r] : d[r + 4], 16);
#pragma unroll
                    for (int r = 0; r < 2; ++r) d[r] = (b3 ? d[r + 2] : d[r]) + __shfl_xor_sync(0xffffffffu, b3 ? d[r] : d[r + 2], 8);
                    float sv = (b2 ? d[1] : d[0]) + __shfl_xor_sync(0xffffffffu, b2 ? d[0] : d[1], 4);
                    sv += __shfl_xor_sync(0xffffffffu, sv, 2);
                    sv += __shfl_xor_sync(0xffffffffu, sv, 1);
                    const int q = wid + NW * (g + (lane >> 2));   // the row of lanes 4 r .. 4 r + 3
                    float inv = 0.0f;
                    if (g + (lane >> 2) < RW && q < nrows) {
                        if (!(sv >= 0x1p-120f && sv <= 0x1p120f)) badr = 1;
                        if ((lane & 3) == 0) sm.srow[q] = sv;
                        inv = rcp_approx(sv);
                    }
#pragma unroll
                    for (int r = 0; r < 8; ++r) d[r] = __shfl_sync(0xffffffffu, inv, 4 * r);
#pragma unroll
                    for (int r = 0; r < 8; ++r) {
                        if (g + r < RG) {
                            const float* kr = Kr[g + r < RG ? g + r : 0];
#pragma unroll
                            for (int x = 0; x < M; ++x) S[x] = fmaf(kr[x], d[r], S[x]);
                        } else if (g + r < RW) {
                            const float* kr = sm.K[(g + r - RG) * NW + wid];
#pragma unroll
                            for (int kk = 0; kk < CH; ++kk) {
                                const float4 v = *(const float4*)(kr + 4 * (lane + 32 * kk));
                                S[4 * kk] = fmaf(v.x, d[r], S[4 * kk]);
                                S[4 * kk + 1] = fmaf(v.y, d[r], S[4 * kk + 1]);
                                S[4 * kk + 2] = fmaf(v.z, d[r], S[4 * kk + 2]);
                                S[4 * kk + 3] = fmaf(v.w, d[r], S[4 * kk + 3]);
                            }
                        }
                    }
                }
                // column partials: the upper half of the warps, then the sums with the lower half
                if (__any_sync(0xffffffffu, badr) && lane == 0) sm.bad = 1;
                float* cp = sm.colpart[wid & (NW / 2 - 1)];
                if (wid >= NW / 2) {
#pragma unroll
                    for (int kk = 0; kk < CH; ++kk)
                        *(float4*)(cp + 4 * (lane + 32 * kk)) = make_float4(S[4 * kk], S[4 * kk + 1], S[4 * kk + 2], S[4 * kk + 3]);
                }
                __syncthreads();
                if (wid < NW / 2) {
#pragma unroll
                    for (int kk = 0; kk < CH; ++kk) {
                        float4* o = (float4*)(cp + 4 * (lane + 32 * kk));
                        const float4 q = *o;
                        *o = make_float4(q.x + S[4 * kk], q.y + S[4 * kk + 1], q.z + S[4 * kk + 2], q.w + S[4 * kk + 3]);
                    }
                }
                __syncthreads();
                // the block's sums of the chunk, to every block; all blocks add them in the same
                // order and so hold the same factors and take the same decisions
                float t4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                if (chunk < NC) {
#pragma unroll
                    for (int x = 0; x < NW / 2; ++x) {
                        const float4 q = *(const float4*)(sm.colpart[x] + 4 * chunk);
                        t4[0] += q.x; t4[1] += q.y; t4[2] += q.z; t4[3] += q.w;
                    }
                    if (sm.bad) t4[0] = __int_as_float(0x7fffffff);   // a row sum left the range: every block ends
#pragma unroll
                    for (int r = 0; r < C; ++r)
                        if (r != (int)rank && r % TWINS == twin)
                            cluster_st4(cluster_map(&sm.inbox[par][rank - (rank > r ? 1 : 0)][4 * chunk], r),
                                        make_float4(t4[0], t4[1], t4[2], t4[3]));
                }
                if (C > 1) cluster_sync();
                bool ok = true, within = true;
                if (chunk < NC) {
                    if (C > 1) {
                        float u4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                        for (int r = 0; r < C; ++r) {
                            float4 q = make_float4(t4[0], t4[1], t4[2], t4[3]);
                            if (r != (int)rank) q = *(const float4*)&sm.inbox[par][r - (r > (int)rank ? 1 : 0)][4 * chunk];
                            u4[0] += q.x; u4[1] += q.y; u4[2] += q.z; u4[3] += q.w;
                        }
#pragma unroll
                        for (int e = 0; e < 4; ++e) t4[e] = u4[e];
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (4 * chunk + e >= n) continue;
                        const float Sj = cj[e] * t4[e];
                        ok = ok && Sj > 0.0f && Sj < INFINITY;
                        within = within && fabsf(Sj - 1.0f) <= (float)A.tol;
                        cj[e] = __fdividef(cj[e], Sj);
                    }
                    if (twin == 0) *(float4*)(sm.c + 4 * chunk) = make_float4(cj[0], cj[1], cj[2], cj[3]);
                }
                bad = !__syncthreads_and(ok);
                const bool conv = __syncthreads_and(within) && !bad;
                ++sweeps;
                done = bad || conv || sweeps >= A.max_sweeps;
                if (done && !bad && !conv) capped = true;
            }
            sweeps_all += sweeps;
            if (bad) break;
            // potentials reached at this p, V_j <- V_j - log2 c_j, and the next step's pairs
            const bool last = k + 1 == A.n_p;
            const double f = last ? 1.0 : A.P[k + 1] / p;
            if (chunk < NC) {   // the twins share the chunk's columns
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int j = 4 * chunk + e;
                    if (e % TWINS != twin || j < v0 || j >= v1) continue;
                    const double v = (sm.V[j - v0] - sum_log2((double)cj[e], sm.l2tab, sm.ltab)) * f;
                    sm.V[j - v0] = v;
                    const float vh = (float)v, vl = (float)(v - (double)vh);
                    if (last) {
                        A.V[A.off[inst] + j] = v * kLn2;
                    } else {
                        sm.vhi()[j] = vh;
                        sm.vlo()[j] = vl;
#pragma unroll
                        for (int r = 0; r < C; ++r)
                            if (r != (int)rank) {
                                cluster_st(cluster_map(sm.vhi() + j, r), vh);
                                cluster_st(cluster_map(sm.vlo() + j, r), vl);
                            }
                    }
                }
            }
            if (last) {
                for (int q = tid; q < nrows; q += NT)
                    A.U[A.off[inst] + r0 + q] = ((double)sm.Cr[q] + sum_log2((double)sm.srow[q], sm.l2tab, sm.ltab)) * kLn2;
            }
            sync_all();
        }
        if (rank == 0 && tid == 0) {
            A.sweeps[inst] = sweeps_all;
            A.status[inst] = bad ? -6 : (capped ? 1 : 0);
        }
        sync_all();   // shared state is rewritten by the next instance
    }
}

}  // namespace sa
