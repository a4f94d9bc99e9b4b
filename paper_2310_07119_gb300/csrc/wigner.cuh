// wigner.cuh - Box-Muller normals of the Wigner noise (Eq. sample) in pairs of floats.
//
// GB300's FP64 rate is 1/64 of its FP32 rate, and the sampled field is stored as floats: a logarithm,
// a square root and a sine-cosine in FP64 cost 30 times the write of the value.  Here each of them is
// carried as an unevaluated sum hi + lo of floats, to about 2^-37 relative (far below the 2^-25 of
// the final rounding to float), from exact integer reductions of the Philox words:
//   ln u    u = a / 2^33 with a = 2 c + 1, a = m 2^e, 1 <= m < 2: a tabulated 8-bit reciprocal r of
//           m's interval (top 7 bits), f = m r - 1 exactly as two floats, and the series of
//           log(1 + f), its first two terms as pairs (the table-driven logarithm of Tang, ACM TOMS
//           16, 1990).  Intervals above sqrt 2 are taken for m / 2, so that ln u keeps its relative
//           accuracy as u -> 1;
//   sqrt    Karp's correction of x rsqrt(x) (Karp and Markstein, ACM TOMS 23, 1997);
//   angle   2 pi u: the nearest of 256 directions in integers, the rest by the series of sin and cos,
//           joined by the addition theorems.
// The functions also compile for the host, so their error can be held without a GPU.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace twa {

struct F2 {  // hi + lo
    float hi, lo;
};
constexpr F2 split2(double x) { return F2{(float)x, (float)(x - (double)(float)x)}; }

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
        const F2 a = split2(q == 0 ? c : (q == 1 ? -s : (q == 2 ? -c : s)));
        const F2 b = split2(q == 0 ? s : (q == 1 ? c : (q == 2 ? -s : -c)));
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
        const F2 t = split2(half ? -ce_ln(2.0 * r) : -ce_ln(r));
        w.rec[i].x = (float)r;
        w.rec[i].y = t.hi;
        w.rec[i].z = t.lo;
        w.rec[i].w = half ? 1.f : 0.f;
    }
    return w;
}

#ifdef __CUDA_ARCH__
#define TWA_CLZ(x) __clz((int)(x))
#define TWA_MUL(a, b) __fmul_rn(a, b)  // a product whose rounding error is taken up later: never part of an fma
#else
#define TWA_CLZ(x) ((x) ? __builtin_clz(x) : 32)
#define TWA_MUL(a, b) ((a) * (b))
#endif

// a + b = s + e exactly (Knuth)
__host__ __device__ __forceinline__ F2 two_sum(float a, float b) {
    const float s = a + b, bb = s - a;
    return F2{s, (a - (s - bb)) + (b - bb)};
}
// the same when |a| >= |b| or a = 0 (Dekker)
__host__ __device__ __forceinline__ F2 fast_two_sum(float a, float b) {
    const float s = a + b;
    return F2{s, b - (s - a)};
}
// (a.hi + a.lo) (b.hi + b.lo)
__host__ __device__ __forceinline__ F2 mul22(F2 a, F2 b) {
    const float p = TWA_MUL(a.hi, b.hi);
    return F2{p, fmaf(a.hi, b.hi, -p) + fmaf(a.hi, b.lo, a.lo * b.hi)};
}

// sqrt(-2 ln u), u = (c + 1/2) / 2^32.
__host__ __device__ __forceinline__ F2 bm_radius(uint32_t c, const float4* rec) {
    // a = 2 c + 1 = (1 + F / 2^32) 2^e
    const int n = 31 - TWA_CLZ(c);                   // -1 for c = 0
    const uint32_t F = c ? (((c << (31 - n)) << 1) | (1u << (31 - n))) : 0u;
    const float4 T = rec[F >> 25];
    const float mh = fmaf((float)(F >> 9), 0x1p-23f, 1.f);   // top 24 bits of m, then the last 9
    const float ml = (float)(F & 511u) * 0x1p-32f;
    // m r - 1: both terms exact (|f| < 2^-7, r of 8 bits), then ordered
    const F2 f = two_sum(fmaf(mh, T.x, -1.f), ml * T.x);
    const float fh = f.hi, fl = f.lo;
    // log(1 + f) = f - f^2 / 2 + f^3 (1/3 - f/4 + f^2/5 - f^3/6 + f^4/7)
    const float f2 = TWA_MUL(fh, fh), f2l = fmaf(fh, fh, -f2) + 2.f * fh * fl;
    const float p = fmaf(fh, fmaf(fh, fmaf(fh, fmaf(fh, 1.f / 7.f, -1.f / 6.f), 0.2f), -0.25f), 1.f / 3.f);
    const float tail = fmaf(fh * f2, p, fmaf(-0.5f, f2l, fl));
    const F2 l = fast_two_sum(fh, -0.5f * f2);
    // ln u = E ln 2 + T + log(1 + f); ln 2 as 15 bits (E ln2_hi is exact) and the rest
    const float E = (float)(n + 1 - 33) + T.w;
    const F2 s0 = fast_two_sum(E * 0x1.62e4p-1f, T.y);       // |E ln 2| >= |T| or E = 0
    const F2 s1 = two_sum(s0.hi, l.hi);
    const float lo = ((s0.lo + s1.lo) + (l.lo + tail)) + fmaf(E, 0x1.7f7d1cp-20f, T.z);
    const F2 L = fast_two_sum(s1.hi, lo);
    const float x = -2.f * L.hi, xl = -2.f * L.lo;
#ifdef __CUDA_ARCH__
    const float y = rsqrtf(x);
#else
    const float y = 1.f / sqrtf(x);
#endif
    const float g = TWA_MUL(x, y);
    return F2{g, 0.5f * y * (fmaf(-g, g, x) + xl)};
}

// cos and sin of 2 pi u, u = (c + 1/2) / 2^32.
__host__ __device__ __forceinline__ void bm_direction(uint32_t c, const float4* dir, F2& co, F2& si) {
    // a = 2 c + 1 units of 2 pi / 2^33: the nearest multiple of 2^25 units, |rest| <= 2^24 (exact in a float)
    const uint32_t j = (c + (1u << 23)) >> 24;               // 0..255, and 0 again past the last (wraps)
    const float rest = (float)(2 * (int32_t)(c - (j << 24)) + 1);
    const float4 D = dir[(c + (1u << 23) < c) ? 0 : j];
    const float kh = 0x1.921fb6p-31f, kl = -0x1.777a5cp-56f; // 2 pi / 2^33
    const float dh = TWA_MUL(rest, kh), dl = fmaf(rest, kh, -dh) + rest * kl;
    const float d2 = TWA_MUL(dh, dh);
    const float d2l = fmaf(dh, dh, -d2) + 2.f * dh * dl;
    // sin d = dh + sl, cos d = 1 + ch + cl
    const float sl = fmaf(dh * d2, fmaf(d2, 1.f / 120.f, -1.f / 6.f), dl);
    const float ch = -0.5f * d2;
    const float cl = fmaf(d2 * d2, fmaf(d2, -1.f / 720.f, 1.f / 24.f), -0.5f * d2l);
    auto turn = [&](float ah, float al, float bh, float bl) {  // a cos d + b sin d
        const float p = TWA_MUL(bh, dh);
        const float pl = fmaf(bh, dh, -p) + fmaf(bh, sl, bl * dh);
        const float q = TWA_MUL(ah, ch);
        const float ql = fmaf(ah, ch, -q) + ah * cl;
        const F2 s = two_sum(ah, p);
        const F2 t = two_sum(s.hi, q);
        return fast_two_sum(t.hi, (s.lo + t.lo) + ((al + pl) + ql));
    };
    co = turn(D.x, D.y, -D.z, -D.w);
    si = turn(D.z, D.w, D.x, D.y);
}

// (a.hi + a.lo) + (b.hi + b.lo), rounded to float once more than exactly
__host__ __device__ __forceinline__ float add22_round(F2 a, F2 b) {
    const F2 s = two_sum(a.hi, b.hi);
    return s.hi + (s.lo + (a.lo + b.lo));
}

}  // namespace twa
