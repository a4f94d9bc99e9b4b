// plain_f64.cu - the FP64 path (complex128): the batched split step of Sec. III.B.2, Eq. mft_normed,
// with every value held and computed in 64 bits.
//
// GB300 runs FP64 at 1/64 of its FP32 rate, so every kernel here is bound by FP64 issue, not by memory:
// what counts is the number of FP64 instructions per value and that all SMs have work.
//   * Line transforms are Stockham radix-4 (a radix-2 stage first when log2 N is odd) of butterflies
//     a +- w b in six fused multiply-adds (a + w b, then 2 a - (a + w b)): 3 instructions per value and
//     radix-2 level instead of 4.  Four values per thread, stages exchanged through shared memory.
//   * A stream's density and potential are real, so two lines of it along the last axis share one complex
//     transform and the other axes run over the half field of N / 2 + 1 planes; the kick, the kinetic
//     phase, the density and 1/k^2 are part of the transform passes.  (Two streams as the real and the
//     imaginary part of one field take as many operations, but a stream that is not finite, or much larger,
//     then spoils its partner: here every stream has the same bits whatever the others of its batch hold.)
//   * All streams of a batch run in each launch.  One launch per stream and operation left most SMs
//     idle: 100 steps of 32 streams of 256 cells took 25,000 launches and 186 ms.
//   * A 1D field stays on one SM for a whole run (k64_run1d), a stream per CTA.
// Measured before and after (one GB300): 100 steps of 32 streams of 256 cells, moments every 10,
// 182.6 -> 1.04 ms; 2 steps of one 128^3 stream and its classical field 9.27 -> 4.22 ms.  (Two streams in one
// transform: 4.18; 32^3 x 16, 50 steps 10.7 ms against 11.1 now, but 512^2 x 8, 20 steps 20.2 against 18.5 and
// 16^3 x 3, 200 steps 21.7 against 18.6.)  A warp's FP64 instruction occupies its scheduler's unit for about
// 100 cycles whatever its active lanes (from the times of 8 to 2048 cells), which is what is left in both.
#include <cuda_runtime.h>

#include "kernels.h"
#include "reduce.cuh"

namespace twa {

__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}

// (a, b) <- (a + w b, a - w b)
__device__ __forceinline__ void bfly(double2& a, double2& b, double2 w) {
    const double2 p = make_double2(fma(w.x, b.x, fma(-w.y, b.y, a.x)), fma(w.x, b.y, fma(w.y, b.x, a.y)));
    b = make_double2(fma(2.0, a.x, -p.x), fma(2.0, a.y, -p.y));
    a = p;
}
__device__ __forceinline__ void bfly1(double2& a, double2& b) {
    const double2 d = make_double2(a.x - b.x, a.y - b.y);
    a = make_double2(a.x + b.x, a.y + b.y);
    b = d;
}

// Radix-4 butterfly with twiddles w1, w2 = w1^2 (conjugated by the caller for an inverse), outputs in order.
template <bool TW>
__device__ __forceinline__ void radix4(double2 (&v)[4], double2 w1, double2 w2, bool inv) {
    if constexpr (TW) {
        bfly(v[0], v[2], w2);
        bfly(v[1], v[3], w2);
        bfly(v[0], v[1], w1);
        bfly(v[2], v[3], inv ? make_double2(-w1.y, w1.x) : make_double2(w1.y, -w1.x));
    } else {
        bfly1(v[0], v[2]);
        bfly1(v[1], v[3]);
        v[3] = inv ? make_double2(-v[3].y, v[3].x) : make_double2(v[3].y, -v[3].x);
        bfly1(v[0], v[1]);
        bfly1(v[2], v[3]);
    }
    // v = outputs 0, 2, 1, 3
    const double2 t = v[1];
    v[1] = v[2];
    v[2] = t;
}

// Shared-memory slot of element i: one 16-byte slot of padding per 8 (the first stages store with
// strides of two and four elements).
__device__ __forceinline__ int pad64(int i) { return i + (i >> 3); }
__host__ __device__ constexpr int line64(int n) { return n + n / 8 + 1; }

// Transform of one line of N = 2^lg values by N / 4 threads: thread j holds elements j + r N / 4, r < 4,
// before and after.  a and b: two exchange lines of line64(N), used in turn by every exchange of a kernel
// (a line is written again only behind the barrier of the exchange in between, so each exchange has
// one barrier); every thread of the CTA takes part.
__device__ __forceinline__ void fft64(double2 (&v)[4], int j, int N, int lg, bool inv, double2*& a, double2*& b,
                                      const double2* __restrict__ tw) {
    auto root = [&](int e) {
        double2 w = __ldg(&tw[e]);
        if (inv) w.y = -w.y;
        return w;
    };
    const int q = N / 4;
    auto exchange = [&](int d0, int d1, int d2, int d3) {
        a[pad64(d0)] = v[0];
        a[pad64(d1)] = v[1];
        a[pad64(d2)] = v[2];
        a[pad64(d3)] = v[3];
        __syncthreads();
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r] = a[pad64(j + r * q)];
        double2* t = a;
        a = b;
        b = t;
    };
    int ls = 0;  // log2 of the sub-transform length ns
    if (lg & 1) {  // radix 2: the butterflies j and j + N / 4
        bfly1(v[0], v[2]);
        bfly1(v[1], v[3]);
        exchange(2 * j, 2 * (j + q), 2 * j + 1, 2 * (j + q) + 1);
        ls = 1;
    }
#pragma unroll 1
    for (; ls < lg; ls += 2) {
        const int ns = 1 << ls, k = j & (ns - 1);
        if (ls == 0) radix4<false>(v, make_double2(1.0, 0.0), make_double2(1.0, 0.0), inv);
        else radix4<true>(v, root(k << (lg - 2 - ls)), root(k << (lg - 1 - ls)), inv);
        if (ls + 2 < lg) {
            const int d = (j - k) * 4 + k;
            exchange(d, d + ns, d + 2 * ns, d + 3 * ns);
        }
    }
}

// z exp(-i theta).  Up to 1/4 sin and cos are their Taylor sums (next terms below 1e-17 relative);
// beyond, theta is reduced mod 2 pi in FP64.  sincos alone took three times the instructions.
__device__ __forceinline__ double2 kick64(double2 z, double th) {
    double s, c;
    if (fabs(th) <= 0.25) {
        const double t = th * th;
        s = fma(t, fma(t, fma(t, fma(t, fma(t, -1.0 / 39916800.0, 1.0 / 362880.0), -1.0 / 5040.0), 1.0 / 120.0), -1.0 / 6.0), 1.0) * th;
        c = fma(t, fma(t, fma(t, fma(t, fma(t, fma(t, 1.0 / 479001600.0, -1.0 / 3628800.0), 1.0 / 40320.0), -1.0 / 720.0),
                                     1.0 / 24.0), -0.5), 1.0);
    } else {
        const double two_pi = 6.283185307179586476925286766559;
        sincos(th - two_pi * rint(th / two_pi), &s, &c);
    }
    return make_double2(fma(z.x, c, z.y * s), fma(z.y, c, -z.x * s));
}

// One axis of a pass: a CTA owns L lines of N = 2^lg values, N / 4 threads a line (power-of-two grids).
struct Axis64 {
    int N, lg, L;
    int S;                       // stride of the axis
    long long lines, cells;      // lines and cells of one field
    const double2* tw;           // exp(-2 pi i m / N)
    const double2* ph;           // exp(-i hbar k^2 dt / 2) / N
};

struct Line64 {
    int j;
    long long at;   // first element of the line in its field
    int step;       // element distance of this thread's four values
    bool act;
    double2 *a, *b;
};
__device__ __forceinline__ Line64 line_of(const Axis64& x) {
    extern __shared__ double2 sm64[];
    Line64 l;
    const int q = x.N / 4;
    // consecutive threads walk along a contiguous line, across the lines of a strided axis
    const int k = x.S == 1 ? threadIdx.x / q : threadIdx.x % x.L;
    l.j = x.S == 1 ? threadIdx.x % q : threadIdx.x / x.L;
    long long id = (long long)blockIdx.x * x.L + k;
    l.act = id < x.lines;
    if (!l.act) id = x.lines - 1;   // partial tiles of small grids run on a clamped line and store nothing
    l.at = x.S == 1 ? id * x.N : (id % x.S) + (id / x.S) * x.S * x.N;
    l.at += (long long)l.j * x.S;
    l.step = q * x.S;
    l.a = sm64 + (size_t)k * line64(x.N);
    l.b = l.a + (size_t)x.L * line64(x.N);
    return l;
}
__device__ __forceinline__ void load4(double2 (&v)[4], const double2* f, const Line64& l) {
#pragma unroll
    for (int r = 0; r < 4; ++r) v[r] = f[l.at + (long long)r * l.step];
}
__device__ __forceinline__ void store4(const double2 (&v)[4], double2* f, const Line64& l) {
    if (!l.act) return;
#pragma unroll
    for (int r = 0; r < 4; ++r) f[l.at + (long long)r * l.step] = v[r];
}
__device__ __forceinline__ void fft4(double2 (&v)[4], Line64& l, const Axis64& x, bool inv) {
    fft64(v, l.j, x.N, x.lg, inv, l.a, l.b, x.tw);
}
__device__ __forceinline__ void drift4(double2 (&v)[4], Line64& l, const Axis64& x) {
    fft4(v, l, x, false);
#pragma unroll
    for (int r = 0; r < 4; ++r) v[r] = zmul(v[r], __ldg(&x.ph[l.j + r * (x.N / 4)]));
    fft4(v, l, x, true);
}

// Slot blockIdx.y of a pass: kick with the potential V that k64_potential left, then, if drift, the axis'
// kinetic factor (rows: a row's cells have one index on the last axis, so V is all real or all imaginary parts).
__global__ void __launch_bounds__(512) k64_kick_drift(Axis64 x, double2* psi, const double2* __restrict__ W,
                                                       long long wcells, double kick, int drift) {
    Line64 l = line_of(x);
    double2 v[4];
    double2* f = psi + (long long)blockIdx.y * x.cells;
    const int upper = l.at >= x.cells / 2;
    const double* V = reinterpret_cast<const double*>(W + (long long)blockIdx.y * wcells) + upper;
    const long long at = l.at - upper * (x.cells / 2);
    load4(v, f, l);
#pragma unroll
    for (int r = 0; r < 4; ++r) v[r] = kick64(v[r], kick * __ldg(&V[2 * (at + (long long)r * l.step)]));
    if (drift) drift4(v, l, x);
    store4(v, f, l);
}

__global__ void __launch_bounds__(512) k64_drift(Axis64 x, double2* psi) {
    Line64 l = line_of(x);
    double2 v[4];
    double2* f = psi + (long long)blockIdx.y * x.cells;
    load4(v, f, l);
    drift4(v, l, x);
    store4(v, f, l);
}

// Last axis of slot blockIdx.y, lines l and l + S / 2 at once (x.lines = S / 2): the axis' kinetic factor (if
// drift), then both lines' densities a and b, transformed as a + i b and taken apart by their symmetry,
//   2 A_k = w_k + conj w_-k,   2 B_k = -i (w_k - conj w_-k),
// into the half field W of N / 2 + 1 planes (the factor 2 is undone by the Poisson multiplier).
__global__ void __launch_bounds__(512) k64_drift_rho(Axis64 x, double2* psi, double2* __restrict__ W, long long wcells,
                                                      int drift) {
    Line64 l = line_of(x);
    double2 v[4], w[4];
    const long long other = x.S / 2;
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        double2* f = psi + (long long)blockIdx.y * x.cells + h * other;
        load4(v, f, l);
        if (drift) {
            drift4(v, l, x);
            store4(v, f, l);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const double d = fma(v[r].x, v[r].x, v[r].y * v[r].y);
            if (h) w[r].y = d;
            else w[r].x = d;
        }
    }
    fft4(w, l, x, false);
    const int q = x.N / 4;
#pragma unroll
    for (int r = 0; r < 4; ++r) l.a[pad64(l.j + r * q)] = w[r];
    __syncthreads();
    if (!l.act) return;
    double2* o = W + (long long)blockIdx.y * wcells + l.at;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        if (r == 2 && l.j > 0) break;   // k = j + r N / 4 up to N / 2
        const double2 c = l.a[pad64((x.N - l.j - r * q) & (x.N - 1))];
        o[(long long)r * l.step] = make_double2(w[r].x + c.x, w[r].y - c.y);
        o[(long long)r * l.step + other] = make_double2(w[r].y + c.y, c.x - w[r].x);
    }
}

// The way back, in place: lines l and l + S / 2 of the half field to the real potentials V of both lines, cells k
// and k + N / 2 as the parts of W's element k (so that every line stays within its own elements, all of which its
// threads have read before the first exchange's barrier).
__global__ void __launch_bounds__(512) k64_potential(Axis64 x, double2* W, long long wcells) {
    Line64 l = line_of(x);
    double2* f = W + (long long)blockIdx.y * wcells + l.at;
    const long long other = x.S / 2;
    double2 v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int k = l.j + r * (x.N / 4);
        const bool conj = k > x.N / 2, real = k == 0 || k == x.N / 2;
        const long long e = (long long)((conj ? x.N - k : k) - l.j) * x.S;
        const double2 a = f[e], b = f[e + other];
        v[r] = real ? make_double2(a.x, b.x)
                    : (conj ? make_double2(a.x + b.y, b.x - a.y) : make_double2(a.x - b.y, a.y + b.x));
    }
    fft4(v, l, x, true);
    if (!l.act) return;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        f[(long long)r * l.step] = make_double2(v[r].x, v[r + 2].x);
        f[(long long)r * l.step + other] = make_double2(v[r].y, v[r + 2].y);
    }
}

// One field src -> dst (which may be the same): forward (mode 0), inverse (1), or forward, Poisson
// multiplier mulc / k^2 (0 at k = 0), inverse (2).
__global__ void __launch_bounds__(512) k64_field(Axis64 x, const double2* src, double2* dst, int mode, int lx, int lxy,
                                                  const double* __restrict__ kx, const double* __restrict__ ky,
                                                  const double* __restrict__ kz, double mulc) {
    Line64 l = line_of(x);
    double2 v[4];
    load4(v, src + (long long)blockIdx.y * x.cells, l);
    fft4(v, l, x, mode == 1);
    if (mode == 2) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const long long e = l.at + (long long)r * l.step;
            const double k2 = __ldg(&kx[e & ((1 << lx) - 1)]) + __ldg(&ky[(e >> lx) & ((1 << (lxy - lx)) - 1)]) +
                              __ldg(&kz[e >> lxy]);
            const double m = k2 > 0.0 ? mulc / k2 : 0.0;
            v[r] = make_double2(v[r].x * m, v[r].y * m);
        }
        fft4(v, l, x, true);
    }
    store4(v, dst + (long long)blockIdx.y * x.cells, l);
}

// One line of 2^LG values for a whole run: V values per thread (2: radix 2; 4: radix 4 with a radix-2 stage
// first when LG is odd), its twiddles in registers.  An exchange of up to 32 threads needs no CTA barrier.
template <int LG, int V>
struct Line1D {
    static constexpr int N = 1 << LG, TH = N / V;
    static constexpr int FIRST = V == 4 && (LG & 1);               // radix-2 stage before the radix-4 ones
    static constexpr int STEP = V == 2 ? 1 : 2;                     // levels per stage
    static constexpr int STAGES = (LG - FIRST) / STEP;
    static constexpr int NTW = V == 2 ? STAGES : 2 * STAGES;
    double2 w[NTW];
    double2 *a, *b;
    int j;
    __device__ __forceinline__ void init(int j_, double2* sm, const double2* __restrict__ tw) {
        j = j_;
        a = sm;
        b = sm + line64(N);
#pragma unroll
        for (int s = 0; s < STAGES; ++s) {
            const int ls = FIRST + s * STEP, k = j & ((1 << ls) - 1);
            if constexpr (V == 2) {
                w[s] = tw[k << (LG - 1 - ls)];
            } else {
                w[2 * s] = tw[k << (LG - 2 - ls)];
                w[2 * s + 1] = tw[k << (LG - 1 - ls)];
            }
        }
    }
    __device__ __forceinline__ void exchange(double2 (&v)[V], const int (&d)[V]) {
#pragma unroll
        for (int r = 0; r < V; ++r) a[pad64(d[r])] = v[r];
        if constexpr (TH <= 32) __syncwarp(TH == 32 ? 0xffffffffu : (1u << (TH & 31)) - 1u);
        else __syncthreads();
#pragma unroll
        for (int r = 0; r < V; ++r) v[r] = a[pad64(j + r * TH)];
        double2* t = a;
        a = b;
        b = t;
    }
    template <bool INV>
    __device__ __forceinline__ void transform(double2 (&v)[V]) {
        auto root = [&](int i) { return INV ? make_double2(w[i].x, -w[i].y) : w[i]; };
        if constexpr (FIRST) {
            bfly1(v[0], v[2]);
            bfly1(v[1], v[3]);
            exchange(v, {2 * j, 2 * (j + TH), 2 * j + 1, 2 * (j + TH) + 1});
        }
#pragma unroll
        for (int s = 0; s < STAGES; ++s) {
            const int ls = FIRST + s * STEP, ns = 1 << ls, k = j & (ns - 1);
            if constexpr (V == 2) {
                if (s == 0) bfly1(v[0], v[1]);
                else bfly(v[0], v[1], root(s));
                const int d = (j - k) * 2 + k;
                if (s + 1 < STAGES) exchange(v, {d, d + ns});
            } else {
                if (ls == 0) radix4<false>(v, w[0], w[0], INV);
                else radix4<true>(v, root(2 * s), root(2 * s + 1), INV);
                const int d = (j - k) * 4 + k;
                if (s + 1 < STAGES) exchange(v, {d, d + ns, d + 2 * ns, d + 3 * ns});
            }
        }
    }
};

// A whole 1D run of one stream (slot blockIdx.x) on one SM: KDK steps with adjacent half kicks merged,
// and at the start and after every out_every steps the synchronized field's |psi|^2, Re psi and Im psi
// per cell (the classical slot: |psi|^2) into partial sums that k_finish_run1d adds over the streams.
// Bound by FP64 issue per scheduler, so up to 256 cells two values per thread keep all four schedulers
// at work (256 x 32: 17.5 us a step against 19.9 with four); batches that fill them anyway take four
// (256 x 500: 41 us against 63).  Twiddles and multipliers stay in registers and the length is a template
// parameter: 100 steps of 32 streams of 256 cells 1.55 -> 1.04 ms.
template <int LG, int V>
__global__ void __launch_bounds__((1 << LG) / V) k64_run1d(double2* psi, const double2* __restrict__ tw,
                                                           const double2* __restrict__ ph, const double* __restrict__ k2,
                                                           double mulc, double kick, int n_out, int out_every, int n_real,
                                                           double* part, double* part_cl, double* part_bad) {
    constexpr int N = 1 << LG;
    extern __shared__ double2 sm64[];
    const int j = threadIdx.x, q = N / V, slot = blockIdx.x;
    Line1D<LG, V> ln;
    ln.init(j, sm64, tw);
    double2* f = psi + (long long)slot * N;
    double2 v[V], p[V];
    double m[V], pot[V];
#pragma unroll
    for (int r = 0; r < V; ++r) {
        v[r] = f[j + r * q];
        p[r] = ph[j + r * q];
        const double k = k2[j + r * q];
        m[r] = k > 0.0 ? mulc / k : 0.0;
    }
    auto poisson = [&]() {
        double2 w[V];
#pragma unroll
        for (int r = 0; r < V; ++r) w[r] = make_double2(fma(v[r].x, v[r].x, v[r].y * v[r].y), 0.0);
        ln.template transform<false>(w);
#pragma unroll
        for (int r = 0; r < V; ++r) w[r] = make_double2(w[r].x * m[r], w[r].y * m[r]);
        ln.template transform<true>(w);
#pragma unroll
        for (int r = 0; r < V; ++r) pot[r] = w[r].x;
    };
    auto output = [&](int o, double kk) {
        if (!part) return;
        int bad = 0;
        double* pp = part + ((long long)o * n_real + slot - 1) * 3 * N;
#pragma unroll
        for (int r = 0; r < V; ++r) {
            const int g = j + r * q;
            const double d = fma(v[r].x, v[r].x, v[r].y * v[r].y);
            if (slot == 0) {
                part_cl[(long long)o * N + g] = d;
                continue;
            }
            const double2 z = kk != 0.0 ? kick64(v[r], kk * pot[r]) : v[r];
            pp[g] = d;
            pp[N + g] = z.x;
            pp[2 * N + g] = z.y;
            bad += (!isfinite(z.x) || !isfinite(z.y)) ? 1 : 0;
        }
        int all = __syncthreads_count(bad > 0);
        if constexpr (V > 1) all += __syncthreads_count(bad > 1);
        if constexpr (V > 2) all += __syncthreads_count(bad > 2) + __syncthreads_count(bad > 3);
        if (slot > 0 && j == 0) part_bad[(long long)o * n_real + slot - 1] = (double)all;
    };
    poisson();
    output(0, 0.0);
#pragma unroll 1
    for (int o = 1; o <= n_out; ++o) {
#pragma unroll 1
        for (int s = 0; s < out_every; ++s) {
            const double kk = (o == 1 && s == 0) ? 0.5 * kick : kick;
#pragma unroll
            for (int r = 0; r < V; ++r) v[r] = kick64(v[r], kk * pot[r]);
            ln.template transform<false>(v);
#pragma unroll
            for (int r = 0; r < V; ++r) v[r] = zmul(v[r], p[r]);
            ln.template transform<true>(v);
            poisson();
        }
        output(o, 0.5 * kick);
    }
    if (n_out == 0) return;
#pragma unroll
    for (int r = 0; r < V; ++r) f[j + r * q] = kick64(v[r], 0.5 * kick * pot[r]);
}

// Per-cell sums over the streams, in slot order: acc = (sum |psi|^2, sum re, sum im).
__global__ void k64_moments_accum(const double2* __restrict__ psi, long long cells, int n_slots, double* acc, double* bad) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < cells; e += (long long)gridDim.x * blockDim.x) {
        double m = 0.0, x = 0.0, y = 0.0;
        int nb = 0;
#pragma unroll 4
        for (int s = 1; s < n_slots; ++s) {
            const double2 z = psi[(long long)s * cells + e];
            m += z.x * z.x + z.y * z.y;
            x += z.x;
            y += z.y;
            nb += (!isfinite(z.x) || !isfinite(z.y)) ? 1 : 0;
        }
        acc[e] = m;
        acc[cells + e] = x;
        acc[2 * cells + e] = y;
        if (nb) atomicAdd(bad, (double)nb);
    }
}

// acc2 (+)= sums of |a_k|^2 and |a_k|^4 over n spectra, in order.
__global__ void k64_modes_accum(const double2* __restrict__ spec, long long cells, int n, double anorm2, int first,
                                double* acc2) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < cells; e += (long long)gridDim.x * blockDim.x) {
        double s2 = first ? 0.0 : acc2[e], s4 = first ? 0.0 : acc2[cells + e];
#pragma unroll 4
        for (int s = 0; s < n; ++s) {
            const double2 z = spec[(long long)s * cells + e];
            const double a2 = anorm2 * (z.x * z.x + z.y * z.y);
            s2 += a2;
            s4 += a2 * a2;
        }
        acc2[e] = s2;
        acc2[cells + e] = s4;
    }
}

__global__ void k64_moments_finish(const double* acc, const double* acc2, const double2* psi0, long long cells, int n_real,
                                   double weyl, double* rho_mean, double* psi_mean, double* rho_cl, double* nk_mean,
                                   double* nk_var, double* part_r, double* part_m, const double* bad) {
    const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    double vr[NP_REAL] = {0, 0, 0, 0, 0, 0};
    double vm[NP_MODES] = {0, 0};
    const double inv = 1.0 / n_real;
    if (g < cells) {
        const double m2 = acc[g] * inv, pr = acc[cells + g] * inv, pi = acc[2 * cells + g] * inv;
        const double2 z0 = psi0[g];
        const double cl = z0.x * z0.x + z0.y * z0.y;
        const double rm = m2 - weyl;
        if (rho_mean) rho_mean[g] = rm;
        if (psi_mean) {
            psi_mean[2 * g] = pr;
            psi_mean[2 * g + 1] = pi;
        }
        if (rho_cl) rho_cl[g] = cl;
        vr[0] = m2 - (pr * pr + pi * pi);
        vr[1] = (rm - cl) * (rm - cl);
        vr[2] = cl * cl;
        vr[3] = m2;
        vr[4] = cl;
        vr[5] = (g == 0) ? *bad : 0.0;
        if (acc2) {
            const double a2 = acc2[g] * inv, a4 = acc2[cells + g] * inv;
            const double nk = a2 - 0.5;
            if (nk_mean) nk_mean[g] = nk;
            if (nk_var) nk_var[g] = a4 - a2 - nk * nk;
            vm[0] = nk;
        }
    }
    block_reduce_store<NP_REAL>(vr, part_r);
    if (part_m) block_reduce_store<NP_MODES>(vm, part_m);
}

// ---------------------------------------------------------------------------------------------
// Host side.
namespace {

int ilog2(int v) {
    int r = 0;
    while ((1 << r) < v) ++r;
    return r;
}
int ew_blocks(long long n) {
    const long long b = (n + 255) / 256;
    return (int)(b < 152 * 16 ? b : 152 * 16);
}

// Lines per CTA: 256 threads for short lines, eight lines (128 bytes of a strided access) up to 256
// cells, then as many as 512 threads (128 registers each) hold.
int lines64(int N) { return N <= 128 ? 1024 / N : 2048 / N; }

Axis64 axis64(const Geom64& g, const Tables64& t, int a) {
    Axis64 x{};
    x.N = g.n[a];
    x.lg = ilog2(x.N);
    x.L = lines64(x.N);
    x.S = 1;
    for (int b = 0; b < a; ++b) x.S *= g.n[b];
    x.cells = g.cells;
    x.lines = g.cells / x.N;
    x.tw = t.tw[a];
    x.ph = t.ph[a];
    return x;
}
unsigned tiles64(const Axis64& x) { return (unsigned)((x.lines + x.L - 1) / x.L); }
int threads64(const Axis64& x) { return x.L * x.N / 4; }
size_t smem64(const Axis64& x) { return 2 * (size_t)x.L * line64(x.N) * sizeof(double2); }

// 2048 cells in a CTA: two exchange buffers of 36 KB
int prepare64() {
    for (const void* k : {(const void*)k64_kick_drift, (const void*)k64_drift, (const void*)k64_drift_rho,
                          (const void*)k64_field, (const void*)k64_potential})
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 80 * 1024) != cudaSuccess) return -3;
    if (cudaFuncSetAttribute(k64_run1d<11, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 80 * 1024) != cudaSuccess) return -3;
    return 0;
}

// cells: of the field, or of the half field of a real one
void field64(const Geom64& g, const Tables64& t, int a, const double2* src, double2* dst, int n, int mode, double mulc,
             long long cells, cudaStream_t st, long long* nl) {
    Axis64 x = axis64(g, t, a);
    x.cells = cells;
    x.lines = cells / x.N;
    const int lx = ilog2(g.n[0]);
    k64_field<<<dim3(tiles64(x), (unsigned)n), threads64(x), smem64(x), st>>>(x, src, dst, mode, lx, lx + ilog2(g.n[1]),
                                                                              t.k2[0], t.k2[1], t.k2[2], mulc);
    ++*nl;
}

// The Poisson solve of n half fields between the transforms of the last axis.
void poisson64(const Geom64& g, const Tables64& t, double2* W, int n, double mulc, cudaStream_t st, long long* nl) {
    const long long wc = f64_half_cells(g);
    if (g.dim == 3) field64(g, t, 1, W, W, n, 0, 0.0, wc, st, nl);
    field64(g, t, 0, W, W, n, 2, mulc, wc, st, nl);
    if (g.dim == 3) field64(g, t, 1, W, W, n, 1, 0.0, wc, st, nl);
}

}  // namespace

int f64_prepare() { return prepare64(); }

int launch_f64_steps(double2* psi, double2* W, int w_slots, int n_slots, const Geom64& g, const Tables64& t, double mulc,
                     double kick, int n_steps, cudaStream_t st, long long* nl) {
    const long long wc = f64_half_cells(g);
    const Axis64 x0 = axis64(g, t, 0);
    Axis64 xl = axis64(g, t, g.dim - 1);
    xl.lines /= 2;   // two at once
    for (int s0 = 0; s0 < n_slots; s0 += w_slots) {
        double2* f = psi + (size_t)s0 * g.cells;
        const unsigned ns = (unsigned)(n_slots - s0 < w_slots ? n_slots - s0 : w_slots);
        auto rho = [&](int drift) {
            k64_drift_rho<<<dim3(tiles64(xl), ns), threads64(xl), smem64(xl), st>>>(xl, f, W, wc, drift);
            poisson64(g, t, W, (int)ns, 0.5 * mulc, st, nl);
            k64_potential<<<dim3(tiles64(xl), ns), threads64(xl), smem64(xl), st>>>(xl, W, wc);
            *nl += 2;
        };
        auto kicks = [&](double k, int drift) {
            k64_kick_drift<<<dim3(tiles64(x0), ns), threads64(x0), smem64(x0), st>>>(x0, f, W, wc, k, drift);
            ++*nl;
        };
        rho(0);
        for (int s = 0; s < n_steps; ++s) {
            kicks(s == 0 ? 0.5 * kick : kick, 1);
            if (g.dim == 3) {
                const Axis64 xm = axis64(g, t, 1);
                k64_drift<<<dim3(tiles64(xm), ns), threads64(xm), smem64(xm), st>>>(xm, f);
                ++*nl;
            }
            rho(1);
        }
        kicks(0.5 * kick, 0);
    }
    return 0;
}

int launch_f64_run1d(double2* psi, int n_slots, const Geom64& g, const Tables64& t, double mulc, double kick, int n_out,
                     int out_every, double* part, double* part_cl, double* part_bad, cudaStream_t st, long long* nl) {
    auto go = [&](auto kernel, int threads) {
        const size_t sm = 2 * (size_t)line64(g.n[0]) * sizeof(double2);
        kernel<<<n_slots, threads, sm, st>>>(psi, t.tw[0], t.ph[0], t.k2[0], mulc, kick, n_out, out_every, n_slots - 1,
                                             part, part_cl, part_bad);
    };
    // from two CTAs per SM on the FP64 units are busy without the second warp of a value pair
    const bool many = n_slots > 2 * 152;
    switch (g.n[0]) {
        case 8: go(k64_run1d<3, 2>, 4); break;
        case 16: go(k64_run1d<4, 2>, 8); break;
        case 32: go(k64_run1d<5, 2>, 16); break;
        case 64: go(k64_run1d<6, 2>, 32); break;
        case 128: many ? go(k64_run1d<7, 4>, 32) : go(k64_run1d<7, 2>, 64); break;
        case 256: many ? go(k64_run1d<8, 4>, 64) : go(k64_run1d<8, 2>, 128); break;
        case 512: go(k64_run1d<9, 4>, 128); break;
        case 1024: go(k64_run1d<10, 4>, 256); break;
        default: go(k64_run1d<11, 4>, 512); break;
    }
    ++*nl;
    return 0;
}

int launch_f64_moments_accum(const double2* psi, long long cells, int n_slots, double* acc, double* bad, cudaStream_t st,
                             long long* nl) {
    k64_moments_accum<<<ew_blocks(cells), 256, 0, st>>>(psi, cells, n_slots, acc, bad);
    ++*nl;
    return 0;
}
int launch_f64_modes(const double2* psi, double2* spec, int spec_fields, int n_slots, const Geom64& g, const Tables64& t,
                     double anorm2, double* acc2, cudaStream_t st, long long* nl) {
    for (int s = 1; s < n_slots; s += spec_fields) {
        const int n = n_slots - s < spec_fields ? n_slots - s : spec_fields;
        for (int a = 0; a < g.dim; ++a)
            field64(g, t, a, a == 0 ? psi + (size_t)s * g.cells : spec, spec, n, 0, 0.0, g.cells, st, nl);
        k64_modes_accum<<<ew_blocks(g.cells), 256, 0, st>>>(spec, g.cells, n, anorm2, s == 1, acc2);
        ++*nl;
    }
    return 0;
}
int launch_f64_moments_finish(const double* acc, const double* acc2, const double2* psi0, long long cells, int n_real,
                              double weyl, double dV, double q_offset, double* rho_mean, double* psi_mean,
                              double* rho_cl, double* nk_mean, double* nk_var, double* part_r, double* part_m,
                              const double* bad, double* scalars, int* err_word, cudaStream_t st, long long* nl) {
    const int nb = (int)((cells + 255) / 256);
    k64_moments_finish<<<nb, 256, 0, st>>>(acc, acc2, psi0, cells, n_real, weyl, rho_mean, psi_mean, rho_cl, nk_mean,
                                            nk_var, part_r, acc2 ? part_m : nullptr, bad);
    ++*nl;
    launch_finish_scalars(part_r, nb, part_m, acc2 ? nb : 0, dV, q_offset, scalars, err_word, st);
    ++*nl;
    return 0;
}

}  // namespace twa
