// wigner.cuh - Box-Muller normals of the Wigner noise (Eq. sample) in pairs of floats.
//
// GB300's FP64 rate is 1/64 of its FP32 rate, and the sampled field is stored as floats: a logarithm,
// a square root and a sine-cosine in FP64 cost 30 times the write of the value.  Here each of them is
// carried as an unevaluated sum hi + lo of floats, the radius to 2^-40.4 relative and the directions to 2^-36.6
// (over all 2^32 words; tests/test_wigner_host.py), from exact integer reductions of the Philox words:
//   ln u    u = a / 2^33 with a = 2 c + 1, a = m 2^e, 1 <= m < 2: a tabulated 8-bit reciprocal r of
//           m's interval (top 7 bits), f = m r - 1 exactly as two floats, and the series of
//           log(1 + f), its first two terms as pairs (the table-driven logarithm of Tang, ACM TOMS
//           16, 1990).  Intervals above sqrt 2 are taken for m / 2, so that ln u keeps its relative
//           accuracy as u -> 1;
//   sqrt    Karp's correction of x rsqrt(x) (Karp and Markstein, ACM TOMS 23, 1997);
//   angle   2 pi u: the nearest of 256 directions in integers, the rest by the series of sin and cos,
//           joined by the addition theorems.
// The arithmetic is written once for a lane type V: float, also on the host, so that its error can be held
// without a GPU, and float2 on the GPU, two values at once in packed FP32 (half the issue slots).
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "fft_engine.cuh"

namespace twa {

template <class V>
struct Pair {  // hi + lo
    V hi, lo;
};
constexpr Pair<float> split2(double x) { return Pair<float>{(float)x, (float)(x - (double)(float)x)}; }

// Tables, formed at compile time in double and split into float pairs (their remainders below 2^-49).
struct WignerTables {
    float4 dir[256];  // cos (hi, lo), sin (hi, lo) of 2 pi j / 256
    float4 rec[128];  // r, -ln r - ln 2 [m / 2 taken] (hi, lo), 1 if m / 2 is taken
};
constexpr double ce_ln(double x) {  // 1/2 <= x <= 2: 2 atanh((x - 1) / (x + 1))
    const double z = (x - 1.0) / (x + 1.0);
    double s = 0.0;
    for (int k = 61; k >= 1; k -= 2) s = s * z * z + 1.0 / k;
    return 2.0 * z * s;
}
constexpr double ce_trig(double x, bool sine) {  // Taylor, |x| <= pi / 4
    double t = sine ? x : 1.0, sum = t;
    for (int k = sine ? 3 : 2; k <= 24; k += 2) {
        t *= -x * x / (k * (k - 1.0));
        sum += t;
    }
    return sum;
}
constexpr WignerTables make_wigner_tables() {
    WignerTables w{};
    const double pi = 3.14159265358979323846;
    for (int j = 0; j < 256; ++j) {
        const int q = ((j + 32) / 64) % 4;          // nearest quarter turn
        const double d = pi * (j - 64 * ((j + 32) / 64)) / 128.0;
        const double c = ce_trig(d, false), s = ce_trig(d, true);
        const Pair<float> a = split2(q == 0 ? c : (q == 1 ? -s : (q == 2 ? -c : s)));
        const Pair<float> b = split2(q == 0 ? s : (q == 1 ? c : (q == 2 ? -s : -c)));
        w.dir[j].x = a.hi;
        w.dir[j].y = a.lo;
        w.dir[j].z = b.hi;
        w.dir[j].w = b.lo;
    }
    for (int i = 0; i < 128; ++i) {
        // the reciprocal of the interval's middle in 1/256ths; 1 and 1/2 at the ends, where ln is small
        int k = (int)(256.0 / (1.0 + (i + 0.5) / 128.0) + 0.5);
        if (i == 0) k = 256;
        if (i == 127) k = 128;
        const bool half = i >= 53;                   // 1 + 53 / 128 = sqrt 2
        const double r = k / 256.0;
        const Pair<float> t = split2(half ? -ce_ln(2.0 * r) : -ce_ln(r));
        w.rec[i].x = (float)r;
        w.rec[i].y = t.hi;
        w.rec[i].z = t.lo;
        w.rec[i].w = half ? 1.f : 0.f;
    }
    return w;
}

#define TWA_HD __host__ __device__ __forceinline__
#ifdef __CUDA_ARCH__
#define TWA_CLZ(x) __clz((int)(x))
// never part of an fma: the rounding errors of these are taken up later
TWA_HD float vadd(float a, float b) { return __fadd_rn(a, b); }
TWA_HD float vsub(float a, float b) { return __fsub_rn(a, b); }
TWA_HD float vmul(float a, float b) { return __fmul_rn(a, b); }
TWA_HD float vrsqrt(float a) { return rsqrtf(a); }
#else
#define TWA_CLZ(x) ((x) ? __builtin_clz(x) : 32)
TWA_HD float vadd(float a, float b) { return a + b; }
TWA_HD float vsub(float a, float b) { return a - b; }
TWA_HD float vmul(float a, float b) { return a * b; }
TWA_HD float vrsqrt(float a) { return 1.f / sqrtf(a); }
#endif
TWA_HD float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return f2_add(a, b); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return f2_sub(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return f2_mul(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return f2_fma(a, b, c); }
__device__ __forceinline__ float2 vrsqrt(float2 a) { return make_float2(rsqrtf(a.x), rsqrtf(a.y)); }
template <class V>
TWA_HD V vset(float c) {
    if constexpr (sizeof(V) == sizeof(float)) return c;
    else return V{c, c};
}
TWA_HD float vneg(float a) { return -a; }
TWA_HD float2 vneg(float2 a) { return float2{-a.x, -a.y}; }

// a + b = s + e exactly (Knuth)
template <class V>
TWA_HD Pair<V> two_sum(V a, V b) {
    const V s = vadd(a, b), bb = vsub(s, a);
    return {s, vadd(vsub(a, vsub(s, bb)), vsub(b, bb))};
}
// the same when |a| >= |b| or a = 0 (Dekker)
template <class V>
TWA_HD Pair<V> fast_two_sum(V a, V b) {
    const V s = vadd(a, b);
    return {s, vsub(b, vsub(s, a))};
}
// (a.hi + a.lo) (b.hi + b.lo)
template <class V>
TWA_HD Pair<V> mul22(Pair<V> a, Pair<V> b) {
    const V p = vmul(a.hi, b.hi);
    return {p, vadd(vfma(a.hi, b.hi, vneg(p)), vfma(a.hi, b.lo, vmul(a.lo, b.hi)))};
}

// The integer reductions of one word c (u = (c + 1/2) / 2^32), as floats.
struct RadiusWord {  // u = a / 2^33, a = 2 c + 1 = (1 + F / 2^32) 2^e
    float mh, ml, E;  // top 24 bits of m and the last 9; e - 33
    float4 T;         // table entry
};
TWA_HD RadiusWord radius_word(uint32_t c, const float4* rec) {
    const int n = 31 - TWA_CLZ(c);                   // -1 for c = 0
    const uint32_t F = c ? (((c << (31 - n)) << 1) | (1u << (31 - n))) : 0u;
    RadiusWord w;
    w.T = rec[F >> 25];
    w.mh = vfma((float)(F >> 9), 0x1p-23f, 1.f);
    w.ml = (float)(F & 511u) * 0x1p-32f;
    w.E = (float)(n + 1 - 33) + w.T.w;
    return w;
}
struct DirectionWord {  // angle = table direction + rest 2 pi / 2^33
    float rest;
    float4 D;
};
TWA_HD DirectionWord direction_word(uint32_t c, const float4* dir) {
    // a = 2 c + 1 units of 2 pi / 2^33: the nearest multiple of 2^25 units, |rest| <= 2^24 (exact in a float)
    const uint32_t j = (c + (1u << 23)) >> 24;       // 0..255, and 0 again past the last (wraps)
    return {(float)(2 * (int32_t)(c - (j << 24)) + 1), dir[j]};
}

// sqrt(-2 ln u) from m = mh + ml, the table's r and -ln r (th + tl), and E.
template <class V>
TWA_HD Pair<V> bm_radius(V mh, V ml, V r, V th, V tl, V E) {
    // m r - 1: both terms exact (|f| < 2^-7, r of 8 bits), then ordered
    const Pair<V> f = two_sum(vfma(mh, r, vset<V>(-1.f)), vmul(ml, r));
    // log(1 + f) = f - f^2 / 2 + f^3 (1/3 - f/4 + f^2/5 - f^3/6 + f^4/7)
    const V f2 = vmul(f.hi, f.hi), f2l = vfma(vadd(f.hi, f.hi), f.lo, vfma(f.hi, f.hi, vneg(f2)));
    const V p = vfma(f.hi, vfma(f.hi, vfma(f.hi, vfma(f.hi, vset<V>(1.f / 7.f), vset<V>(-1.f / 6.f)), vset<V>(0.2f)),
                                vset<V>(-0.25f)), vset<V>(1.f / 3.f));
    const V tail = vfma(vmul(f.hi, f2), p, vfma(vset<V>(-0.5f), f2l, f.lo));
    const Pair<V> l = fast_two_sum(f.hi, vmul(vset<V>(-0.5f), f2));
    // ln u = E ln 2 - ln r + log(1 + f); ln 2 as 15 bits (E ln2_hi is exact) and the rest
    const Pair<V> s0 = fast_two_sum(vmul(E, vset<V>(0x1.62e4p-1f)), th);   // |E ln 2| >= |ln r| or E = 0
    const Pair<V> s1 = two_sum(s0.hi, l.hi);
    const V lo = vadd(vadd(vadd(s0.lo, s1.lo), vadd(l.lo, tail)), vfma(E, vset<V>(0x1.7f7d1cp-20f), tl));
    const Pair<V> L = fast_two_sum(s1.hi, lo);
    const V x = vmul(vset<V>(-2.f), L.hi), xl = vmul(vset<V>(-2.f), L.lo);
    const V y = vrsqrt(x);
    const V g = vmul(x, y);
    return {g, vmul(vmul(vset<V>(0.5f), y), vadd(vfma(vneg(g), g, x), xl))};
}

// cos and sin of the angle: directions (ch + cl, sh + sl) of the table turned by rest 2 pi / 2^33.
template <class V>
TWA_HD void bm_direction(V rest, V ch, V cl, V sh, V sl, Pair<V>& co, Pair<V>& si) {
    const V kh = vset<V>(0x1.921fb6p-31f), kl = vset<V>(-0x1.777a5cp-56f);  // 2 pi / 2^33
    const V dh = vmul(rest, kh), dl = vfma(rest, kl, vfma(rest, kh, vneg(dh)));
    const V d2 = vmul(dh, dh);
    const V d2l = vfma(vadd(dh, dh), dl, vfma(dh, dh, vneg(d2)));
    // sin d = dh + ds, cos d = 1 + qh + ql
    const V ds = vfma(vmul(dh, d2), vfma(d2, vset<V>(1.f / 120.f), vset<V>(-1.f / 6.f)), dl);
    const V qh = vmul(vset<V>(-0.5f), d2);
    const V ql = vfma(vmul(d2, d2), vfma(d2, vset<V>(-1.f / 720.f), vset<V>(1.f / 24.f)), vmul(vset<V>(-0.5f), d2l));
    auto turn = [&](V ah, V al, V bh, V bl) {  // a cos d + b sin d
        const V p = vmul(bh, dh);
        const V pl = vadd(vfma(bh, dh, vneg(p)), vfma(bh, ds, vmul(bl, dh)));
        const V q = vmul(ah, qh);
        const V e = vfma(ah, ql, vfma(ah, qh, vneg(q)));
        const Pair<V> s = two_sum(ah, p);
        const Pair<V> t = two_sum(s.hi, q);
        return fast_two_sum(t.hi, vadd(vadd(s.lo, t.lo), vadd(vadd(al, pl), e)));
    };
    co = turn(ch, cl, vneg(sh), vneg(sl));
    si = turn(sh, sl, ch, cl);
}

}  // namespace twa
