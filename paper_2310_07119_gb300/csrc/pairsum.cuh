// pairsum.cuh - running sums of floats as unevaluated pairs (the moment kernels).
#pragma once
#include "fft_engine.cuh"

namespace twa {

// Running sum of floats carried as an unevaluated pair hi + lo ("double-float"): each addition's
// rounding error is recovered exactly (Knuth's two-sum) and the pair is renormalized (Dekker's
// fast two-sum), so the sum keeps about 48 significant bits.  The moment kernels accumulate in
// this form because this part's FP64 rate is 1/64 of its FP32 rate: FP64 adds would make them
// compute-bound at several times their memory time.  Results are finished in FP64.
struct DF {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float a) {
        const float s = hi + a;
        const float bp = s - hi;
        float e = (hi - (s - bp)) + (a - bp);  // hi + a = s + e exactly
        e += lo;
        hi = s + e;
        lo = e - (hi - s);
    }
    // add a * a exactly (the product's rounding error recovered with an fma)
    __device__ __forceinline__ void add_sq(float a) {
        const float p = a * a;
        const float q = fmaf(a, a, -p);
        add(p);
        lo += q;
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// Two float-pair sums at once (DF, in packed two-lane FP32: half the issue slots).  add_sq adds a * a,
// its product unrounded (both uses inside an fma).
struct DF2 {
    float2 hi = make_float2(0.f, 0.f), lo = make_float2(0.f, 0.f);
    __device__ __forceinline__ void finish(float2 s, float2 bp, float2 abp) {
        const float2 e = f2_add(f2_add(f2_sub(hi, f2_sub(s, bp)), abp), lo);
        hi = f2_add(s, e);
        lo = f2_sub(e, f2_sub(hi, s));
    }
    __device__ __forceinline__ void add(float2 a) {
        const float2 s = f2_add(hi, a), bp = f2_sub(s, hi);
        finish(s, bp, f2_sub(a, bp));
    }
    __device__ __forceinline__ void add_sq(float2 a) {
        const float2 s = f2_fma(a, a, hi), bp = f2_sub(s, hi);
        finish(s, bp, f2_fma(a, a, make_float2(-bp.x, -bp.y)));
    }
    // a to the first sum, a * a exactly to the second (DF::add and DF::add_sq)
    __device__ __forceinline__ void add_with_square(float a) {
        const float p = __fmul_rn(a, a);
        add(make_float2(a, p));
        lo.y += fmaf(a, a, -p);
    }
    __device__ __forceinline__ double x() const { return (double)hi.x + (double)lo.x; }
    __device__ __forceinline__ double y() const { return (double)hi.y + (double)lo.y; }
};

}  // namespace twa
