// log2pair.cuh -- float-pair arithmetic for the exponent p log2 w - C_i - V_j of the
// per-step matrices (the step kernel and the Newton path): exact two-sum and a log2 of
// integer weights accurate to about 2^-40 from a 256-entry shared table and a short series.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "sa_internal.h"

namespace sa {

// Row references of K from scaled row potentials lie up to cs log2 n above the row maxima (cs:
// the ratio of the p values); beyond this many powers of two the maxima are taken instead,
// while the largest entries of K are still far above the FP32 underflow.
constexpr double kMaxRefShift = 64.0;

constexpr int kLog2Tab = 32768;   // weights below this take the shared-table logarithm

// s + err = a + b exactly (Knuth's two-sum; no FMA contraction is possible here)
__device__ __forceinline__ float two_sum(float a, float b, float* err) {
    const float s = a + b;
    const float bb = s - a;
    *err = (a - (s - bb)) + (b - bb);
    return s;
}

// the sum of two unevaluated pairs (to about 2^-47)
__device__ __forceinline__ void pair_add(float& hi, float& lo, float h2, float l2) {
    float e;
    hi = two_sum(hi, h2, &e);
    lo = (lo + l2) + e;
}

// Shared table for log2 of a weight: entry j (the top 8 mantissa bits of m in [1, 2)) holds
// g_j = 1 / (1 + (j + 0.5)/256) rounded to 9 significant bits and -log2(g_j) as a float pair.
__device__ __forceinline__ float4 log2_tab_entry(int j) {
    const double c = 1.0 + (j + 0.5) / 256.0;
    const double g = ldexp(rint(ldexp(1.0 / c, 8)), -8);   // 9 significant bits (value in (0.5, 1))
    const double t = -log2(g);
    const float th = (float)t;
    return make_float4((float)g, th, (float)(t - (double)th), 0.0f);
}

// log2 w (0 < w < 2^15) as an unevaluated float pair, accurate to about 2^-40 (2^-38.7 at most): with
// w = 2^e m, m g_j is exact (15 + 9 significant bits), so r = m g_j - 1 is exact and
// |r| < 2^-7.4; log2 w = e + (-log2 g_j) + log2(1 + r), the last from its series with the
// leading product r log2(e) split exactly.
__device__ __forceinline__ float2 log2_pair(int w, const float4* tab) {
    const unsigned bits = __float_as_uint((float)w);
    const int e = (int)(bits >> 23) - 127;
    const float4 t = tab[(bits >> 15) & 0xFFu];
    const float m = __uint_as_float((bits & 0x7FFFFFu) | 0x3F800000u);
    const float r = fmaf(m, t.x, -1.0f);
    const float l2eh = 1.4426950216293335f, l2el = 1.925963033500011e-08f;   // log2(e) as a pair
    const float ph = r * l2eh;
    const float pe = fmaf(r, l2eh, -ph);
    // ln(1 + r) / r - 1 = -r/2 + r^2/3 - r^3/4 + r^4/5 - r^5/6 (next term below 2^-48)
    const float poly = r * (-0.5f + r * (0.333333343f + r * (-0.25f + r * (0.2f + r * -0.166666672f))));
    const float small = fmaf(r, l2el, pe) + ph * poly;
    float e1, e2;
    const float s1 = two_sum((float)e, t.y, &e1);
    const float s2 = two_sum(s1, ph, &e2);
    return make_float2(s2, ((e1 + e2) + t.z) + small);
}

// log2 of s = hi + lo (hi a normal number) as a pair, to about 2^-46 of an exponent up to 31 (rms; 2^-43.6
// at most): the reduction of sum_log2 in FP32 (m g - 1 is exact: 24 + 8 bits of which the
// leading 8 cancel)
__device__ __forceinline__ float2 pair_log2(float hi, float lo, const float4* tab) {
    const unsigned bits = __float_as_uint(hi);
    const int e = (int)(bits >> 23) - 127;
    const float d = hi - 1.0f;
    const bool near = fabsf(d) < 0x1p-8f;
    const float4 t = tab[(bits >> 15) & 0xffu];
    const float m = __uint_as_float((bits & 0x7fffffu) | 0x3f800000u);
    const float scale = __uint_as_float((unsigned)(min(max(-e, -126), 126) + 127) << 23);
    const float r = near ? d : fmaf(m, t.x, -1.0f);
    const float rl = near ? lo : lo * scale * t.x;
    const float b0 = near ? 0.0f : (float)e, b1 = near ? 0.0f : t.y, b2 = near ? 0.0f : t.z;
    const float l2eh = 1.4426950216293335f, l2el = 1.925963033500011e-08f;   // log2(e) as a pair
    // ln(1 + r + rl) = a + tail, the square split exactly, the cubic and the rest below 2^-23
    const float q = r * r, qe = fmaf(r, r, -q);
    float e0, e1, e2;
    const float a = two_sum(r, -0.5f * q, &e0);
    const float cub = q * r * (0.333333343f + r * (-0.25f + r * (0.2f + r * -0.166666672f)));
    const float tail = (e0 - 0.5f * qe) + (fmaf(rl, q - r, rl) + cub);
    const float ph = a * l2eh;
    const float pe = fmaf(tail, l2eh, fmaf(a, l2el, fmaf(a, l2eh, -ph)));
    const float s1 = two_sum(b1, ph, &e1);   // both below 1: the exponent's addition rounds last
    const float s2 = two_sum(b0, s1, &e2);
    return make_float2(s2, ((e1 + b2) + pe) + e2);
}

// the same for |a| >= |b|
__device__ __forceinline__ float fast_two_sum(float a, float b, float* err) {
    const float s = a + b;
    *err = b - (s - a);
    return s;
}

// log2 of a weight of 2^15 .. 2^31 - 1 as a pair: pair_log2's reduction of the weight as a float and an
// exact remainder (r exact, |r| < 2^-7.4; rl below 2^-24), every term kept to 2^-49 and
// the pair normalised, so that only the rounding of its second part is left: rms 2^-46.2, at
// most 2^-44.96 over 20 million weights (an FP64 logarithm split into a pair 2^-44.91, pair_log2
// 2^-43.6).  About 80 FP32 instructions; the FP64 logarithm is about 45 FP64 instructions, at two
// of them per clock and SM: 0.4 ms of 2.8 at n = 2047, growing as n^2.
__device__ __forceinline__ float2 wide_log2(int w, const float4* tab) {
    const float hi = (float)w;                                   // up to 2^31
    const float lo = (float)(int)((unsigned)w - (unsigned)hi);
    const unsigned bits = __float_as_uint(hi);
    const int ex = (int)(bits >> 23) - 127;
    const float4 t = tab[(bits >> 15) & 0xffu];
    const float m = __uint_as_float((bits & 0x7fffffu) | 0x3f800000u);
    const float r = fmaf(m, t.x, -1.0f);
    const float rl = lo * __uint_as_float((unsigned)(127 - ex) << 23) * t.x;   // exact
    const float l2eh = 1.4426950216293335f, l2el = 1.925963033500011e-08f;   // log2(e) as a pair
    const float th3 = 0.333333343f, tl3 = -9.934108e-09f;                      // 1/3 as a pair
    float e1, e2, e3, e4;
    // r - r^2 / 2 = a + e0 - qe / 2; r^3 (1/3 + s) = ch + cl
    const float q = __fmul_rn(r, r), qe = fmaf(r, r, -q);
    const float a = fmaf(-0.5f, q, r), e0 = fmaf(-0.5f, q, r - a);
    const float c = __fmul_rn(q, r), ce = fmaf(qe, r, fmaf(q, r, -c));
    const float s = r * fmaf(r, fmaf(r, -0.166666672f, 0.2f), -0.25f);
    const float ch = __fmul_rn(c, th3), cl = fmaf(c, s, fmaf(ce, th3, fmaf(c, tl3, fmaf(c, th3, -ch))));
    // ln(1 + r + rl) = a + th + tl, with rl / (1 + r) - rl^2 / 2 for the remainder
    const float th = two_sum(ch, rl, &e3);
    const float tl = e3 + (cl + (e0 + fmaf(rl, q - (r + fmaf(0.5f, rl, c)), -0.5f * qe)));
    const float ph = __fmul_rn(a, l2eh), pe = fmaf(a, l2eh, -ph);
    const float xh = __fmul_rn(th, l2eh);
    const float xl = fmaf(th, l2el, fmaf(tl, l2eh, fmaf(a, l2el, pe)) + fmaf(th, l2eh, -xh));
    const float s1 = two_sum(t.y, ph, &e1);
    const float s2 = fast_two_sum((float)ex, s1, &e2);
    float z = two_sum(e1, xh, &e3);
    z = two_sum(z, t.z, &e4);
    float zl = xl + (e3 + e4);
    const float v = two_sum(e2, z, &e3);
    zl += e3;
    const float v2 = v + zl;
    const float h = fast_two_sum(s2, v2, &e4);
    return make_float2(h, e4 + ((v - v2) + zl));
}
// out of line: inlined in the unrolled loops over a row it made the evaluation longer for all
// weights (n = 20000, int16: 1.86 against 1.75 ms)
static __device__ __noinline__ float2 wide_log2_call(int w, const float4* tab) { return wide_log2(w, tab); }

// log2 of a positive integer weight as a float pair, from the shared table: the short series for
// the int16 range, the longer one above it.
__device__ __forceinline__ float2 wlog2(const float4* stab, int w) {
    return w < kLog2Tab ? log2_pair(w, stab) : wide_log2_call(w, stab);
}

// The same for four weights (-inf, 0 for one that is not positive): the four chains of a
// wide logarithm overlap, and one call serves them.
struct WideLog4 {
    float4 h, l;
};
static __device__ __noinline__ WideLog4 wide_log4(int w0, int w1, int w2, int w3, const float4* tab) {
    const float2 a = wide_log2(w0, tab), b = wide_log2(w1, tab), c = wide_log2(w2, tab), d = wide_log2(w3, tab);
    return {make_float4(a.x, b.x, c.x, d.x), make_float4(a.y, b.y, c.y, d.y)};
}
__device__ __forceinline__ void wlog2_4(const float4* stab, const int w[4], float lh[4], float ll[4]) {
    WideLog4 x{};
    const bool wide = max(max(w[0], w[1]), max(w[2], w[3])) >= kLog2Tab;
    if (wide) x = wide_log4(w[0], w[1], w[2], w[3], stab);
    const float xh[4] = {x.h.x, x.h.y, x.h.z, x.h.w}, xl[4] = {x.l.x, x.l.y, x.l.z, x.l.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        float2 p = make_float2(-INFINITY, 0.0f);
        if (w[e] > 0) p = w[e] < kLog2Tab ? log2_pair(w[e], stab) : make_float2(xh[e], xl[e]);
        lh[e] = p.x;
        ll[e] = p.y;
    }
}

// 2^(p log2 w - V_j - m) with the operands as float pairs (p = ph + pl): the large leading
// parts cancel exactly (two-product, two-sums), the small ones are added after; the exponent
// x is then exact to about 2^-24 |x|
__device__ __forceinline__ float pair_exp2(float ph, float pl, float2 lw, float vh, float vl, float mh, float ml) {
    const float t = ph * lw.x;
    const float te = fmaf(ph, lw.x, -t);
    float e1, e2;
    const float s1 = two_sum(t, -vh, &e1);
    const float s2 = two_sum(s1, -mh, &e2);
    const float rest = ((te + e1) + e2) + (fmaf(ph, lw.y, pl * lw.x) - vl - ml);
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(s2 + rest));
    return y;
}

// log2 of s > 0 in FP64: the mantissa times a 9-bit reciprocal from the table is 1 + r exactly,
// |r| < 2^-7; near 1 r = s - 1 itself.  ltab[j] = -log2(tab[j].x) in FP64.  One formula for all
// arguments, about 20 FP64 instructions where the library's log2 takes some hundred: GB300 runs
// two of them per clock and SM.
__device__ __forceinline__ double sum_log2(double s, const float4* tab, const double* ltab) {
    const int hi = __double2hiint(s);
    const int e = (hi >> 20) - 1023;
    const int idx = (hi >> 12) & 255;
    const double m = __hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(s));
    const double d = s - 1.0;
    const bool near = fabs(d) < 0x1p-8;
    const double r = near ? d : fma(m, (double)tab[idx].x, -1.0);
    const double base = near ? 0.0 : (double)e + ltab[idx];
    // ln(1 + r) / r up to r^6 (the next term is below 2^-59)
    const double r2 = r * r;
    const double a = fma(r, -0.5, 1.0), b = fma(r, -0.25, 1.0 / 3.0), c = fma(r, -1.0 / 6.0, 0.2);
    const double q = fma(r2, fma(r2, fma(r2, 1.0 / 7.0, c), b), a);
    return fma(r * kLog2e, q, base);
}

}  // namespace sa
