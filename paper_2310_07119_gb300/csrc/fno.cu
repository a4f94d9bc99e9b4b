// fno.cu - Fourier-neural-operator surrogate of the TWA correction spectrum: forward, backward,
// AdamW, with BF16 weights (FP32 master copy) and FP32 accumulation.
//
// Network (features on the grid of Fourier modes of an n^3 field, layout [B][C][n][n][n]):
//   h_0 = P x + p;  z_l = Re A^H (R_l . A h_l) + W_l h_l + b_l;  h_{l+1} = gelu(z_l) (l < L-1);
//   y = Q h_L + q.
// A is the unitary 3D DFT restricted to the frequencies |m_a| < modes on each axis, applied as three
// axis transforms with (2 modes) x n complex matrices; A^H is its adjoint.  R_l holds one complex
// W x W matrix per retained mode.  All reductions (weight gradients, the loss) run in a fixed
// order, so training is bitwise reproducible.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <type_traits>
#include <vector>

#include "reduce.cuh"
#include "tc_gemm.h"
#include "twa.h"

void twa_set_global_error(const std::string& msg);

namespace {

constexpr int kThreads = 256;
constexpr int kPwBlocks = 152 * 2;  // CTAs of the pointwise weight gradient's first stage (and its partials)
constexpr int kMixWgradSmem = 100 * 1024;

int blocks_for(long long n) {
    const long long b = (n + kThreads - 1) / kThreads;
    return (int)(b < 152LL * 64 ? b : 152LL * 64);
}

// Packed two-lane FP32 (sm_100 and later): d = a b + c on both halves, each rounded once.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
        "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
template <int BYTES>
__device__ __forceinline__ void cp_async(void* s, const void* g) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(s)), "l"(g), "n"(BYTES));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N)); }

// out[p][i][q] = sum_j M[i][j] in[p][j][q] (complex M, nout x nin), one axis of the truncated DFT.  INR:
// the input is real; OUTR: only the real part is kept, and added to out if accumulate.
//
// A batched complex matrix product with 30 to 60 FP32 operations a byte: bound by the FP32 units, once
// their operands do not come from shared memory one by one.  A CTA owns AX_COLS columns (p, q) and up
// to 32 outputs; a thread 8 outputs x 4 columns, two outputs to a packed FMA, so that 6 128-bit reads
// of shared memory feed 64 packed FMAs (one thread per column and 16 outputs, an operand read per two
// FMAs, took 5.8 ms of a 128^3 x 2 forward pass of width 32, 16 modes and 4 layers; now 1.9 ms).  The columns' values come in
// double-buffered slices of AX_J rows by cp.async.  The sum of an output runs over j in order.
constexpr int AX_COLS = 128, AX_J = 16, AX_O = 8;
template <bool INR, bool OUTR>
__global__ void __launch_bounds__(128) k_axis(const void* __restrict__ in, const float2* __restrict__ M, void* __restrict__ out,
                                              long long cols, int nin, int nout, long long Q, int accumulate) {
    extern __shared__ __align__(16) float4 axsm[];
    using X = typename std::conditional<INR, float, float2>::type;
    const int og = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ob = blockIdx.y * 4 * AX_O, o0 = ob + og * AX_O;   // this CTA's and this warp's outputs
    float4* Ms = axsm;                                          // [j][pair of outputs] (re0, re1, im0, im1)
    X* Xs = reinterpret_cast<X*>(Ms + (size_t)2 * AX_O * nin);  // [2][AX_J][AX_COLS]
    for (int t = threadIdx.x; t < 2 * AX_O * nin; t += 128) {
        const int pr = t / nin, j = t - pr * nin, i = ob + 2 * pr;
        const float2 a = i < nout ? M[(long long)i * nin + j] : make_float2(0.f, 0.f);
        const float2 b = i + 1 < nout ? M[(long long)(i + 1) * nin + j] : make_float2(0.f, 0.f);
        Ms[j * 2 * AX_O + pr] = make_float4(a.x, b.x, a.y, b.y);
    }
    const long long c0 = (long long)blockIdx.x * AX_COLS;
    // copies: a thread per column where those are contiguous, lanes along j where the axis is (Q = 1)
    const X* src = static_cast<const X*>(in);
    {
        const long long col = min(c0 + threadIdx.x, cols - 1), p = Q == 1 ? 0 : col / Q;
        if (Q != 1) src += p * nin * Q + (col - p * Q);
    }
    auto load = [&](int j0, int buf) {
        X* dst = Xs + buf * AX_J * AX_COLS;
        if (Q != 1) {
#pragma unroll
            for (int jj = 0; jj < AX_J; ++jj)
                if (j0 + jj < nin) cp_async<sizeof(X)>(dst + jj * AX_COLS + threadIdx.x, src + (long long)(j0 + jj) * Q);
        } else {
            const int jj = threadIdx.x % AX_J;
#pragma unroll 4
            for (int c = threadIdx.x / AX_J; c < AX_COLS; c += 128 / AX_J)
                if (j0 + jj < nin)
                    cp_async<sizeof(X)>(dst + jj * AX_COLS + c, src + min(c0 + c, cols - 1) * nin + j0 + jj);
        }
        cp_commit();
    };
    float2 ar[AX_O / 2][4], ai[AX_O / 2][4];
#pragma unroll
    for (int u = 0; u < AX_O / 2; ++u)
#pragma unroll
        for (int c = 0; c < 4; ++c) ar[u][c] = ai[u][c] = make_float2(0.f, 0.f);
    const int slices = (nin + AX_J - 1) / AX_J;
    load(0, 0);
    for (int s = 0; s < slices; ++s) {
        if (s + 1 < slices) {
            load((s + 1) * AX_J, (s + 1) & 1);
            cp_wait<1>();
        } else {
            cp_wait<0>();
        }
        __syncthreads();
        const X* xs = Xs + (size_t)(s & 1) * AX_J * AX_COLS + lane * 4;
        const int nj = min(AX_J, nin - s * AX_J);
        if (o0 < nout)
#pragma unroll 4
        for (int jj = 0; jj < nj; ++jj) {
            const float4* m = Ms + (s * AX_J + jj) * 2 * AX_O + og * (AX_O / 2);
            float2 x[4];
            if constexpr (INR) {
                const float4 v = *reinterpret_cast<const float4*>(xs + jj * AX_COLS);
                x[0].x = v.x;
                x[1].x = v.y;
                x[2].x = v.z;
                x[3].x = v.w;
            } else {
                const float4 v = reinterpret_cast<const float4*>(xs + jj * AX_COLS)[0];
                const float4 w = reinterpret_cast<const float4*>(xs + jj * AX_COLS)[1];
                x[0] = make_float2(v.x, v.y);
                x[1] = make_float2(v.z, v.w);
                x[2] = make_float2(w.x, w.y);
                x[3] = make_float2(w.z, w.w);
            }
#pragma unroll
            for (int u = 0; u < AX_O / 2; ++u) {
                const float4 mm = m[u];
                const float2 mr = make_float2(mm.x, mm.y), mi = make_float2(mm.z, mm.w);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float2 xr = make_float2(x[c].x, x[c].x);
                    if constexpr (INR) {
                        ar[u][c] = fma2(mr, xr, ar[u][c]);
                        ai[u][c] = fma2(mi, xr, ai[u][c]);
                    } else {
                        const float2 xn = make_float2(-x[c].y, -x[c].y), xi = make_float2(x[c].y, x[c].y);
                        ar[u][c] = fma2(mr, xr, fma2(mi, xn, ar[u][c]));
                        if constexpr (!OUTR) ai[u][c] = fma2(mr, xi, fma2(mi, xr, ai[u][c]));
                    }
                }
            }
        }
        __syncthreads();
    }
    if (o0 >= nout) return;
    const long long col = c0 + lane * 4;
    if (!OUTR && (Q & 3) == 0) {  // the four columns are neighbours in memory
        if (col >= cols) return;
        const long long p = col / Q, q = col - p * Q;
#pragma unroll
        for (int u = 0; u < AX_O; ++u) {
            if (o0 + u >= nout) break;
            float4* d = reinterpret_cast<float4*>(static_cast<float2*>(out) + (p * nout + o0 + u) * Q + q);
#pragma unroll
            for (int h = 0; h < 2; ++h)
                d[h] = u & 1 ? make_float4(ar[u / 2][2 * h].y, ai[u / 2][2 * h].y, ar[u / 2][2 * h + 1].y, ai[u / 2][2 * h + 1].y)
                             : make_float4(ar[u / 2][2 * h].x, ai[u / 2][2 * h].x, ar[u / 2][2 * h + 1].x, ai[u / 2][2 * h + 1].x);
        }
        return;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        if (col + c >= cols) break;
        const long long p = Q == 1 ? col + c : (col + c) / Q, q = col + c - p * Q;
#pragma unroll
        for (int u = 0; u < AX_O; ++u) {
            const int i = o0 + u;
            if (i >= nout) break;
            const long long d = (p * nout + i) * Q + q;
            const float re = u & 1 ? ar[u / 2][c].y : ar[u / 2][c].x;
            if constexpr (OUTR) {
                float* o = static_cast<float*>(out);
                o[d] = accumulate ? o[d] + re : re;
            } else {
                static_cast<float2*>(out)[d] = make_float2(re, u & 1 ? ai[u / 2][c].y : ai[u / 2][c].x);
            }
        }
    }
}

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_g(float z) {
    return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// Y[b][o][k] = sum_c W[o][c] X[b][c][k] + bias[o] (+ Y if accumulate); TRANS reads W as [c][o].  What
// follows the map in the network is part of it: EP_GELU also stores gelu(Y) to Z, EP_GRAD stores
// Y gelu'(Z) instead of Y.
//
// Bound by memory (width 32 with EP_GELU: 4 arrays of 128 bytes a position for 1024 FMAs) as long as
// the weights are cheap and enough loads are in flight: a thread holds PW_O outputs of P positions, two
// outputs to a packed FMA, so that a 128-bit read of the weights feeds 2 P of them, eight inputs ahead.
// 32 outputs take two positions: four need 220 registers and leave 8 warps an SM.
// Positions come P to a load when every row starts on 16 bytes (VEC), else one by one, a block apart.  (One position per thread, its inputs
// in local memory, and gelu passes of their own took 5.1 ms of a 128^3 x 2 forward pass; now 2.5 ms.)
enum { EP_NONE = 0, EP_GELU, EP_GRAD };
template <int PW_O, int P, bool TRANS, int EP, bool VEC>
__global__ void __launch_bounds__(128, 4) k_pointwise(const float* __restrict__ X, const __nv_bfloat16* __restrict__ Wt,
                                                   const float* __restrict__ bias, float* Y, float* Z, int B, int cin,
                                                   int cout, long long K, int accumulate) {
    __shared__ __align__(16) float ws[64 * PW_O];   // [c][o] of this block of outputs
    __shared__ float bs[PW_O];
    const int o0 = blockIdx.y * PW_O;
    for (int i = threadIdx.x; i < cin * PW_O; i += 128) {
        const int c = i / PW_O, o = o0 + i % PW_O;
        ws[i] = o < cout ? __bfloat162float(Wt[TRANS ? c * cout + o : o * cin + c]) : 0.f;
    }
    for (int i = threadIdx.x; i < PW_O; i += 128) bs[i] = bias && o0 + i < cout ? bias[o0 + i] : 0.f;
    __syncthreads();
    // positions k0 + u st, u < P
    const long long k0 = blockIdx.x * (128LL * P) + threadIdx.x * (VEC ? P : 1);
    const int st = VEC ? 1 : 128;
    if (k0 >= K) return;
    auto get = [&](const float* p, float (&v)[P]) {
        if constexpr (VEC && P == 4) {
            const float4 t = *reinterpret_cast<const float4*>(p);
            v[0] = t.x;
            v[1] = t.y;
            v[2] = t.z;
            v[3] = t.w;
        } else if constexpr (VEC) {
            const float2 t = *reinterpret_cast<const float2*>(p);
            v[0] = t.x;
            v[1] = t.y;
        } else {
#pragma unroll
            for (int u = 0; u < P; ++u) v[u] = k0 + u * st < K ? p[u * st] : 0.f;
        }
    };
    auto put = [&](float* p, const float (&v)[P]) {
        if constexpr (VEC && P == 4) {
            *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
        } else if constexpr (VEC) {
            *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
        } else {
#pragma unroll
            for (int u = 0; u < P; ++u)
                if (k0 + u * st < K) p[u * st] = v[u];
        }
    };
    for (long long b = blockIdx.z; b < B; b += gridDim.z) {
        const float* x = X + b * cin * K + k0;
        float2 acc[PW_O / 2][P];
#pragma unroll
        for (int o = 0; o < PW_O / 2; ++o)
#pragma unroll
            for (int u = 0; u < P; ++u) acc[o][u] = make_float2(bs[2 * o], bs[2 * o + 1]);
#pragma unroll 8
        for (int c = 0; c < cin; ++c) {
            float v[P];
            get(x + c * K, v);
            const float4* w = reinterpret_cast<const float4*>(ws + c * PW_O);
#pragma unroll
            for (int o = 0; o < PW_O / 4; ++o) {
                const float4 ww = w[o];
#pragma unroll
                for (int u = 0; u < P; ++u) {
                    acc[2 * o][u] = fma2(make_float2(ww.x, ww.y), make_float2(v[u], v[u]), acc[2 * o][u]);
                    acc[2 * o + 1][u] = fma2(make_float2(ww.z, ww.w), make_float2(v[u], v[u]), acc[2 * o + 1][u]);
                }
            }
        }
        // G outputs at a time: their loads first, as the stores may alias them for the compiler
        constexpr int G = PW_O < 8 ? PW_O : 8;
#pragma unroll
        for (int og = 0; og < PW_O; og += G) {
            if (o0 + og >= cout) break;
            float t[G][P], z[G][P];
            const long long at = (b * cout + o0 + og) * K + k0;
#pragma unroll
            for (int o = 0; o < G; ++o)
                if (accumulate && o0 + og + o < cout) get(Y + at + o * K, t[o]);
            if constexpr (EP == EP_GRAD) {
#pragma unroll
                for (int o = 0; o < G; ++o)
                    if (o0 + og + o < cout) get(Z + at + o * K, z[o]);
            }
#pragma unroll
            for (int o = 0; o < G; ++o) {
                if (o0 + og + o >= cout) break;
                float r[P];
#pragma unroll
                for (int u = 0; u < P; ++u) {
                    r[u] = (og + o) & 1 ? acc[(og + o) / 2][u].y : acc[(og + o) / 2][u].x;
                    if (accumulate) r[u] = t[o][u] + r[u];
                    if constexpr (EP == EP_GRAD) r[u] = r[u] * gelu_g(z[o][u]);
                }
                put(Y + at + o * K, r);
                if constexpr (EP == EP_GELU) {
#pragma unroll
                    for (int u = 0; u < P; ++u) r[u] = gelu_f(r[u]);
                    put(Z + at + o * K, r);
                }
            }
        }
    }
}

// Partial sums of dW[o][c] = sum_{b,k} dY[b][o][k] X[b][c][k] and db[o] = sum dY over the chunks of
// positions of CTA blockIdx.x, for outputs and inputs in blocks of 32 (blockIdx.y).  part[o][blk][c],
// c = cin for db; k_pointwise_wgrad_sum adds the blocks in a fixed order.
//
// The 32 x 32 sums sit in the registers of 16 threads (8 x 8 each), and 16 such groups take every
// sixteenth group of four positions of a chunk, copied to shared memory one chunk ahead: 16 128-bit
// reads feed 256 FMAs (one product per two reads took 536 us a call at 64^3 x 4, width 32, 24 times its reads from HBM;
// now 90 us).  Rows are padded so that the eight rows a quarter warp reads lie in distinct banks.
constexpr int WG_CH = 128, WG_LD = WG_CH + 4, WG_SMEM = 2 * 64 * WG_LD * 4;
template <bool VEC>
__global__ void __launch_bounds__(256) k_pointwise_wgrad(const float* __restrict__ dY, const float* __restrict__ X, int B,
                                                         int cin, int cout, long long K, float* __restrict__ part) {
    extern __shared__ __align__(16) float wgsm[];     // two buffers of 32 rows of dY, 32 rows of X
    __shared__ float sb[16][32];
    const int nci = (cin + 31) / 32, o0 = (blockIdx.y / nci) * 32, i0 = (blockIdx.y % nci) * 32;
    const int grp = threadIdx.x / 16, ty = (threadIdx.x % 16) / 4, tx = threadIdx.x % 4;  // rows ty + 4 u, tx + 4 u
    float acc[8][8], ab[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        ab[u] = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) acc[u][w] = 0.f;
    }
    const long long kch = (K + WG_CH - 1) / WG_CH, total = (long long)B * kch;
    // rows past the last output or input stay zero; positions past the last are copied as zeros
    for (int i = threadIdx.x; i < 2 * 64 * WG_LD; i += 256) wgsm[i] = 0.f;
    __syncthreads();
    auto load = [&](long long ch, float* dst) {
        const long long b = ch / kch, k0 = (ch - b * kch) * WG_CH;
        constexpr int E = VEC ? 4 : 1, PER = WG_CH / E;   // floats per copy, copies per row
#pragma unroll 8
        for (int i = threadIdx.x; i < 64 * PER; i += 256) {
            const int row = i / PER, k = (i % PER) * E;
            const bool y = row < 32;
            const int r = y ? o0 + row : i0 + row - 32;
            if (r >= (y ? cout : cin)) continue;
            const bool in = k0 + k < K;
            const float* g = (y ? dY : X) + (b * (y ? cout : cin) + r) * K + (in ? k0 + k : 0);
            asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"((unsigned)__cvta_generic_to_shared(dst + row * WG_LD + k)),
                         "l"(g), "n"(E * 4), "r"(in ? E * 4 : 0));
        }
        cp_commit();
    };
    if (blockIdx.x < total) load(blockIdx.x, wgsm);
    int buf = 0;
    for (long long ch = blockIdx.x; ch < total; ch += gridDim.x, buf ^= 1) {
        if (ch + gridDim.x < total) {
            load(ch + gridDim.x, wgsm + (buf ^ 1) * 64 * WG_LD);
            cp_wait<1>();
        } else {
            cp_wait<0>();
        }
        __syncthreads();
        const float* cur = wgsm + buf * 64 * WG_LD;
#pragma unroll
        for (int g = 0; g < WG_CH / 64; ++g) {
            const float* s = cur + (grp + 16 * g) * 4;
            float4 y[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                y[u] = *reinterpret_cast<const float4*>(s + (ty + 4 * u) * WG_LD);
                if (tx == 0) ab[u] += (y[u].x + y[u].y) + (y[u].z + y[u].w);
            }
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                const float4 x = *reinterpret_cast<const float4*>(s + (32 + tx + 4 * w) * WG_LD);
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    acc[u][w] = fmaf(y[u].w, x.w, fmaf(y[u].z, x.z, fmaf(y[u].y, x.y, fmaf(y[u].x, x.x, acc[u][w]))));
            }
        }
        __syncthreads();
    }
    // the sixteen groups' sums in group order, four rows u at a time (16 x 4 x 32 floats each)
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 8; ++u)
        if (tx == 0) sb[grp][ty + 4 * u] = ab[u];
    const int nb = gridDim.x;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int w = 0; w < 8; ++w) wgsm[(grp * 16 + ty + 4 * u) * 32 + tx + 4 * w] = acc[4 * h + u][w];
        __syncthreads();
        for (int t = threadIdx.x; t < 512; t += 256) {
            float v = 0.f;
#pragma unroll
            for (int g = 0; g < 16; ++g) v += wgsm[g * 512 + t];
            const int o = o0 + 16 * h + t / 32, c = i0 + t % 32;
            if (o < cout && c < cin) part[((long long)o * nb + blockIdx.x) * (cin + 1) + c] = v;
        }
    }
    if (i0 == 0 && threadIdx.x < 32 && o0 + threadIdx.x < cout) {
        float v = 0.f;
#pragma unroll
        for (int g = 0; g < 16; ++g) v += sb[g][threadIdx.x];
        part[((long long)(o0 + threadIdx.x) * nb + blockIdx.x) * (cin + 1) + cin] = v;
    }
}

// dW and db += the blocks' partial sums: a CTA of 128 threads per output o; thread t adds blocks in
// order for its c (a tree over a warp's lanes would read them uncoalesced).
__global__ void k_pointwise_wgrad_sum(const float* __restrict__ part, int cin, int nblk, float* __restrict__ dW,
                                      float* __restrict__ db) {
    // 128 threads: (cin + 1) columns in up to 128 / (cin + 1) slices of the blocks, the slices added in order
    __shared__ float red[128];
    const int o = blockIdx.x, nc = cin + 1, slices = 128 / nc, sl = threadIdx.x / nc, c = threadIdx.x % nc;
    float s = 0.f;
    if (sl < slices)
        for (int i = sl; i < nblk; i += slices) s += part[((long long)o * nblk + i) * nc + c];
    red[threadIdx.x] = s;
    __syncthreads();
    if (sl == 0) {
        for (int u = 1; u < slices; ++u) s += red[u * nc + c];
        if (c < cin) dW[o * cin + c] += s;
        else db[o] += s;
    }
}

// Per retained mode m: Y[b][o] = sum_c R[o][c] S[b][c], or ADJ: dS[b][c] = sum_o conj(R[o][c]) G[b][o] (R
// complex BF16, W x W).  Every R is used once, so the call is bound by reading R (134 MB at 32^3 modes
// and width 32): thread (x, mode) holds one output channel x for MIX_B batch elements, reads its row
// of R four complex numbers at a time (R4; rows of an ADJ product are read across the threads), and
// takes the modes' inputs from shared memory, where a warp's threads read one address.  CTAs of
// MIX_T / W modes.  (R staged in shared memory and read with a 16-way bank conflict, in two CTAs per
// SM, took 356 us a call at 128^3 x 2; now 58 us.)
constexpr int MIX_T = 256, MIX_B = 4;
enum { R_SCALAR = 0, R_COMPLEX, R_FOUR };   // loads of R: its reals, complex numbers, four of them
template <bool ADJ, int RL>
__global__ void __launch_bounds__(MIX_T) k_mix(const float2* __restrict__ S, const __nv_bfloat16* __restrict__ R,
                                               float2* __restrict__ Y, int B, int W, long long Mm, int MB) {
    extern __shared__ float2 mxsm[];
    const int LD = W + 1;                             // padded: the copies walk along the modes
    float2* Ss = mxsm;                                // [min(B, MIX_B)][mode][W]
    float2* Ys = Ss + (size_t)MIX_B * MB * LD;        // the same of the results
    const int x = threadIdx.x % W, mm = threadIdx.x / W, nt = MB * W;
    const long long m0 = (long long)blockIdx.x * MB;
    const int nm = (int)min((long long)MB, Mm - m0);
    for (int b0 = 0; b0 < B; b0 += MIX_B) {
        const int nb = min(MIX_B, B - b0);
        __syncthreads();
        for (int i = threadIdx.x; i < nb * W * MB; i += nt) {
            const int k = i % MB, bc = i / MB;
            if (k < nm) Ss[((bc / W) * MB + k) * LD + bc % W] = S[((long long)b0 * W + bc) * Mm + m0 + k];
        }
        __syncthreads();
        if (mm < nm) {
            float2 acc[MIX_B];
#pragma unroll
            for (int b = 0; b < MIX_B; ++b) acc[b] = make_float2(0.f, 0.f);
            const long long r0 = (m0 + mm) * W * W + (ADJ ? x : (long long)x * W);   // complex elements
            auto step = [&](int c, __nv_bfloat162 q) {
                const float2 w = __bfloat1622float2(q);
                const float rim = ADJ ? -w.y : w.y;
#pragma unroll
                for (int b = 0; b < MIX_B; ++b) {
                    if (b >= nb) break;
                    const float2 v = Ss[(b * MB + mm) * LD + c];
                    acc[b].x = fmaf(w.x, v.x, fmaf(-rim, v.y, acc[b].x));
                    acc[b].y = fmaf(w.x, v.y, fmaf(rim, v.x, acc[b].y));
                }
            };
            if constexpr (RL == R_FOUR) {
                const uint4* r = reinterpret_cast<const uint4*>(R + 2 * r0);
#pragma unroll 4
                for (int c = 0; c < W; c += 4) {
                    const uint4 q = r[c / 4];
                    step(c, *reinterpret_cast<const __nv_bfloat162*>(&q.x));
                    step(c + 1, *reinterpret_cast<const __nv_bfloat162*>(&q.y));
                    step(c + 2, *reinterpret_cast<const __nv_bfloat162*>(&q.z));
                    step(c + 3, *reinterpret_cast<const __nv_bfloat162*>(&q.w));
                }
            } else {
#pragma unroll 8
                for (int c = 0; c < W; ++c) {
                    const long long d = r0 + (ADJ ? (long long)c * W : c);
                    step(c, RL == R_COMPLEX ? reinterpret_cast<const __nv_bfloat162*>(R)[d]
                                            : __nv_bfloat162(R[2 * d], R[2 * d + 1]));
                }
            }
#pragma unroll
            for (int b = 0; b < MIX_B; ++b)
                if (b < nb) Ys[(b * MB + mm) * LD + x] = acc[b];
        }
        __syncthreads();
        for (int i = threadIdx.x; i < nb * W * MB; i += nt) {
            const int k = i % MB, bc = i / MB;
            if (k < nm) Y[((long long)b0 * W + bc) * Mm + m0 + k] = Ys[((bc / W) * MB + k) * LD + bc % W];
        }
    }
}

// dR[m][o][c] += sum_b G[b][o][m] conj(S[b][c][m])   (re/im interleaved in the flat gradient): bound by
// reading and writing dR (2 x 268 MB at 32^3 modes and width 32).  A CTA holds the inputs of MB modes
// in shared memory with the channels side by side, so that threads on consecutive c read distinct
// banks (PAIR: two c and 16 bytes of dR per thread).  With the modes side by side it took 316 us a
// call at 64^3 x 4, width 32, 32^3 modes; now 126 us.
template <bool PAIR>
__global__ void __launch_bounds__(MIX_T) k_mix_wgrad(const float2* __restrict__ G, const float2* __restrict__ S,
                                                     float* __restrict__ dR, int B, int W, long long Mm, int MB) {
    extern __shared__ float2 mxsm[];
    const int LD = W + 1;
    float2* Gs = mxsm;                       // [B][mode][W]
    float2* Ss = Gs + (size_t)B * MB * LD;
    const long long m0 = (long long)blockIdx.x * MB;
    const int nm = (int)min((long long)MB, Mm - m0);
    for (int i = threadIdx.x; i < B * W * MB; i += MIX_T) {
        const int k = i % MB, bc = i / MB;
        if (k < nm) {
            Gs[((bc / W) * MB + k) * LD + bc % W] = G[(long long)bc * Mm + m0 + k];
            Ss[((bc / W) * MB + k) * LD + bc % W] = S[(long long)bc * Mm + m0 + k];
        }
    }
    __syncthreads();
    auto dot = [&](int mm, int o, int c) {
        float2 a = make_float2(0.f, 0.f);
        for (int b = 0; b < B; ++b) {
            const float2 g = Gs[(b * MB + mm) * LD + o], v = Ss[(b * MB + mm) * LD + c];
            a.x = fmaf(g.x, v.x, fmaf(g.y, v.y, a.x));
            a.y = fmaf(g.y, v.x, fmaf(-g.x, v.y, a.y));
        }
        return a;
    };
    if constexpr (PAIR) {
        float4* d = reinterpret_cast<float4*>(dR + 2 * m0 * W * W);
        const int h = W / 2;
#pragma unroll 4
        for (int i = threadIdx.x; i < nm * W * h; i += MIX_T) {
            const int c = i % h, o = (i / h) % W, mm = i / (h * W);
            const float2 p = dot(mm, o, 2 * c), q = dot(mm, o, 2 * c + 1);
            const float4 r = d[i];
            d[i] = make_float4(r.x + p.x, r.y + p.y, r.z + q.x, r.w + q.y);
        }
    } else {
        for (int i = threadIdx.x; i < nm * W * W; i += MIX_T) {
            const float2 p = dot(i / (W * W), (i / W) % W, i % W);
            const long long t = m0 * W * W + i;
            dR[2 * t] += p.x;
            dR[2 * t + 1] += p.y;
        }
    }
}

// The same without shared memory, for batches whose inputs of one mode exceed it.
__global__ void k_mix_wgrad_any(const float2* __restrict__ G, const float2* __restrict__ S, float* __restrict__ dR, int B,
                                int W, long long Mm) {
    const long long total = Mm * W * W;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(t % W), o = (int)((t / W) % W);
        const long long m = t / ((long long)W * W);
        float ar = 0.f, ai = 0.f;
        for (int b = 0; b < B; ++b) {
            const float2 g = G[((long long)b * W + o) * Mm + m];
            const float2 s = S[((long long)b * W + c) * Mm + m];
            ar = fmaf(g.x, s.x, fmaf(g.y, s.y, ar));
            ai = fmaf(g.y, s.x, fmaf(-g.x, s.y, ai));
        }
        dR[2 * t] += ar;
        dR[2 * t + 1] += ai;
    }
}

// MSE: per-block partial sums of (y - t)^2 and dy = 2 (y - t) / n; then a fixed-order final sum.
__global__ void k_mse_part(const float* __restrict__ y, const float* __restrict__ t, long long n, float* __restrict__ dy,
                           double* __restrict__ part) {
    double acc[1] = {0.0};
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float d = y[i] - t[i];
        acc[0] += (double)d * d;
        if (dy) dy[i] = 2.f * d / (float)n;
    }
    twa::block_reduce_store<1>(acc, part);
}
__global__ void k_mse_final(const double* __restrict__ part, int nb, long long n, float* __restrict__ loss) {
    __shared__ double red[256];
    double s = 0.0;
    for (int b = threadIdx.x; b < nb; b += 256) s += part[b];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) *loss = (float)(red[0] / (double)n);
}

// Bound by memory: 30 bytes a parameter, read and written four at a time (268 M parameters: 1.59 ms
// one at a time, now 1.16 ms).
__global__ void k_adamw(float* __restrict__ th, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                        __nv_bfloat16* __restrict__ th16, long long n, float lr, float b1, float b2, float eps, float wd,
                        float c1, float c2) {
    auto one = [&](float& t, float gi, float& mi, float& vi) {
        mi = b1 * mi + (1.f - b1) * gi;
        vi = b2 * vi + (1.f - b2) * gi * gi;
        const float upd = (mi / c1) / (sqrtf(vi / c2) + eps) + wd * t;
        t = t - lr * upd;
    };
    const long long i0 = blockIdx.x * (long long)blockDim.x + threadIdx.x, st = (long long)gridDim.x * blockDim.x;
    for (long long i = i0; i < n / 4; i += st) {
        float4 t = reinterpret_cast<float4*>(th)[i], a = reinterpret_cast<float4*>(m)[i], b = reinterpret_cast<float4*>(v)[i];
        const float4 gi = reinterpret_cast<const float4*>(g)[i];
        one(t.x, gi.x, a.x, b.x);
        one(t.y, gi.y, a.y, b.y);
        one(t.z, gi.z, a.z, b.z);
        one(t.w, gi.w, a.w, b.w);
        reinterpret_cast<float4*>(th)[i] = t;
        reinterpret_cast<float4*>(m)[i] = a;
        reinterpret_cast<float4*>(v)[i] = b;
        reinterpret_cast<__nv_bfloat162*>(th16)[2 * i] = __floats2bfloat162_rn(t.x, t.y);
        reinterpret_cast<__nv_bfloat162*>(th16)[2 * i + 1] = __floats2bfloat162_rn(t.z, t.w);
    }
    for (long long i = n / 4 * 4 + i0; i < n; i += st) {
        one(th[i], g[i], m[i], v[i]);
        th16[i] = __float2bfloat16(th[i]);
    }
}

__global__ void k_to_bf16(const float* __restrict__ a, __nv_bfloat16* __restrict__ b, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        b[i] = __float2bfloat16(a[i]);
}

}  // namespace

// ---------------------------------------------------------------------------------------------
struct twa_fno {
    twa_fno_config cfg{};
    long long n_params = 0;
    // offsets into the flat parameter vector
    long long oP = 0, op = 0, oQ = 0, oq = 0;
    std::vector<long long> oR, oW, ob;
    float* th = nullptr;            // FP32 master
    __nv_bfloat16* th16 = nullptr;  // BF16 copy used by the kernels
    float* grad = nullptr;
    float* am = nullptr;
    float* av = nullptr;
    long long step = 0;
    float2* Mf[3] = {nullptr, nullptr, nullptr};  // forward truncated DFT per axis (2m x n)
    float2* Mi[3] = {nullptr, nullptr, nullptr};  // adjoint (n x 2m)
    // the x-axis (contiguous) contractions as real GEMMs on the tensor cores (tc_gemm.cu):
    // Bf [npf][n]: rows (Re, Im) of the 2m DFT rows; Ba [npa][4m]: per cell the (Re, -Im) of its adjoint row
    float* Bf = nullptr;
    float* Ba = nullptr;
    int npf = 0, npa = 0;
    bool tc_fwd = false, tc_adj = false, tc_on = true;
    int* d_err = nullptr;
    // activations and workspaces for the largest batch seen (held in acts)
    int cap_b = 0;
    std::vector<float*> h, z;   // h[layers] is z[layers - 1]
    std::vector<float2*> s;
    float2* t1 = nullptr;
    float2* t2 = nullptr;
    float2* mixed = nullptr;
    float* dz = nullptr;        // dL/dz of the current layer, and the next one's as it is formed
    float* dz2 = nullptr;
    float* part = nullptr;
    double* lpart = nullptr;
    const float* x_in = nullptr;
    int last_b = 0;
    std::vector<void*> allocs, acts;
    std::string err;
};

namespace {

int ffail(twa_fno* f, int code, const std::string& m) {
    if (f) f->err = m;
    twa_set_global_error(m);
    return code;
}

#define FC(call)                                                                          \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess) return ffail(f, TWA_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

template <class T>
int falloc(twa_fno* f, T** p, size_t n, std::vector<void*>* owner = nullptr) {
    if (cudaMalloc((void**)p, (n ? n : 1) * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return ffail(f, TWA_ENOMEM, "twa_fno: cudaMalloc failed");
    }
    (owner ? owner : &f->allocs)->push_back(*p);
    return 0;
}

long long kcells(const twa_fno* f) { return (long long)f->cfg.grid * f->cfg.grid * f->cfg.grid; }
long long kmodes(const twa_fno* f) {
    const long long m2 = 2LL * f->cfg.modes;
    return m2 * m2 * m2;
}

// Free the activations and workspaces of the largest batch seen, and forget the forward that filled them.
void drop_batch(twa_fno* f) {
    f->cap_b = f->last_b = 0;
    f->x_in = nullptr;
    for (void* p : f->acts) cudaFree(p);
    f->acts.clear();
    f->h.clear();
    f->z.clear();
    f->s.clear();
    f->t1 = f->t2 = f->mixed = nullptr;
    f->dz = f->dz2 = nullptr;
}

// Room for a batch of B.  When it cannot be had the model holds none at all: a backward is refused, and the
// next forward starts afresh.
int ensure_batch(twa_fno* f, int B) {
    if (B <= f->cap_b) return 0;
    drop_batch(f);
    const int L = f->cfg.layers, W = f->cfg.width, n = f->cfg.grid, m2 = 2 * f->cfg.modes;
    const size_t act = (size_t)B * W * kcells(f), modes = (size_t)B * W * kmodes(f);
    const size_t tsz = (size_t)B * W * n * n * (size_t)(m2 > n ? m2 : n);
    f->h.assign(L, nullptr);
    f->z.assign(L, nullptr);
    f->s.assign(L, nullptr);
    int rc = 0;
    auto get = [&](auto** p, size_t count) {
        if (!rc) rc = falloc(f, p, count, &f->acts);
    };
    for (int l = 0; l < L; ++l) get(&f->h[l], act);
    for (int l = 0; l < L; ++l) {
        get(&f->z[l], act);
        get(&f->s[l], modes);
    }
    get(&f->t1, tsz);
    get(&f->t2, tsz);
    get(&f->mixed, modes);
    get(&f->dz, act);
    get(&f->dz2, act);
    if (rc) {
        drop_batch(f);
        return rc;
    }
    f->h.push_back(f->z[L - 1]);
    f->cap_b = B;
    return 0;
}

// Kernel attributes of the current device (at creation).
int fno_prepare() {
    cudaError_t e = cudaSuccess;
    auto set = [&](const void* k, int bytes) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    };
    const int ax = 2 * AX_O * 128 * 16 + 2 * AX_J * AX_COLS * 8;
    set((const void*)k_axis<false, false>, ax);
    set((const void*)k_axis<true, false>, ax);
    set((const void*)k_axis<false, true>, ax);
    set((const void*)k_pointwise_wgrad<true>, WG_SMEM);
    set((const void*)k_pointwise_wgrad<false>, WG_SMEM);
    set((const void*)k_mix_wgrad<true>, kMixWgradSmem);
    set((const void*)k_mix_wgrad<false>, kMixWgradSmem);
    return e == cudaSuccess ? 0 : -3;
}

// One axis contraction of a complex (in_c) or real (in_r) input into a complex (out_c) or real (out_r) output.
void axis_launch(cudaStream_t st, const float2* in_c, const float* in_r, const float2* M, float2* out_c, float* out_r,
                 long long P, int nin, int nout, long long Q, int accumulate) {
    const long long cols = P * Q;
    const dim3 grid((unsigned)((cols + AX_COLS - 1) / AX_COLS), (unsigned)((nout + 4 * AX_O - 1) / (4 * AX_O)));
    const size_t sm = (size_t)2 * AX_O * nin * sizeof(float4) + 2 * AX_J * AX_COLS * (in_r ? sizeof(float) : sizeof(float2));
    if (in_r)
        k_axis<true, false><<<grid, 128, sm, st>>>(in_r, M, out_c, cols, nin, nout, Q, 0);
    else if (out_r)
        k_axis<false, true><<<grid, 128, sm, st>>>(in_c, M, out_r, cols, nin, nout, Q, accumulate);
    else
        k_axis<false, false><<<grid, 128, sm, st>>>(in_c, M, out_c, cols, nin, nout, Q, 0);
}

bool aligned(const void* p, unsigned bytes) { return (reinterpret_cast<uintptr_t>(p) & (bytes - 1)) == 0; }

template <bool ADJ>
void mix_launch(const float2* S, const __nv_bfloat16* R, float2* Y, int B, int W, long long Mm, cudaStream_t st) {
    const int MB = MIX_T / W;   // modes per CTA (W <= 64)
    const size_t sm = (size_t)2 * MIX_B * MB * (W + 1) * sizeof(float2);
    const unsigned nb = (unsigned)((Mm + MB - 1) / MB);
    // the layers' matrices start where the ones before them end: on 16, 4 or 2 bytes
    if (!ADJ && W % 4 == 0 && aligned(R, 16))
        k_mix<ADJ, R_FOUR><<<nb, MB * W, sm, st>>>(S, R, Y, B, W, Mm, MB);
    else if (aligned(R, 4))
        k_mix<ADJ, R_COMPLEX><<<nb, MB * W, sm, st>>>(S, R, Y, B, W, Mm, MB);
    else
        k_mix<ADJ, R_SCALAR><<<nb, MB * W, sm, st>>>(S, R, Y, B, W, Mm, MB);
}

void mix_wgrad_launch(const float2* G, const float2* S, float* dR, int B, int W, long long Mm, cudaStream_t st) {
    const size_t one = (size_t)2 * B * (W + 1) * sizeof(float2);   // one mode
    if (one > (size_t)kMixWgradSmem) {
        k_mix_wgrad_any<<<blocks_for(Mm * W * W), kThreads, 0, st>>>(G, S, dR, B, W, Mm);
        return;
    }
    // eight modes (64-byte segments of the inputs) as far as 48 KB hold them
    const int MB = one * 8 <= 48 * 1024 ? 8 : (one <= 48 * 1024 ? (int)(48 * 1024 / one) : 1);
    const unsigned nb = (unsigned)((Mm + MB - 1) / MB);
    if (W % 2 == 0 && aligned(dR, 16))
        k_mix_wgrad<true><<<nb, MIX_T, one * MB, st>>>(G, S, dR, B, W, Mm, MB);
    else
        k_mix_wgrad<false><<<nb, MIX_T, one * MB, st>>>(G, S, dR, B, W, Mm, MB);
}

// A (truncated forward DFT) of a real [B*W][n][n][n] field into complex [B*W][2m][2m][2m].
void dft_fwd(twa_fno* f, const float* in, float2* out, long long BW, cudaStream_t st) {
    const int n = f->cfg.grid, m2 = 2 * f->cfg.modes;
    // x axis (last): (BW*n*n, n, 1) -> (BW*n*n, 2m, 1); on the tensor cores when the shape allows
    if (!(f->tc_on && f->tc_fwd &&
          twa::tc_gemm(in, BW * n * n, n, n, f->Bf, 2 * m2, f->npf, reinterpret_cast<float*>(f->t1), 2 * m2, 0, f->d_err,
                  2.0, st) == 0))
        axis_launch(st, nullptr, in, f->Mf[2], f->t1, nullptr, BW * n * n, n, m2, 1, 0);
    // y axis: (BW*n, n, 2m) -> (BW*n, 2m, 2m)
    axis_launch(st, f->t1, nullptr, f->Mf[1], f->t2, nullptr, BW * n, n, m2, m2, 0);
    // z axis: (BW, n, 4m^2) -> (BW, 2m, 4m^2)
    axis_launch(st, f->t2, nullptr, f->Mf[0], out, nullptr, BW, n, m2, (long long)m2 * m2, 0);
}

// Re A^H of complex [BW][2m][2m][2m] into a real [BW][n][n][n] field (overwrite or add).
void dft_adj(twa_fno* f, const float2* in, float* out, long long BW, int accumulate, cudaStream_t st) {
    const int n = f->cfg.grid, m2 = 2 * f->cfg.modes;
    axis_launch(st, in, nullptr, f->Mi[0], f->t1, nullptr, BW, m2, n, (long long)m2 * m2, 0);
    axis_launch(st, f->t1, nullptr, f->Mi[1], f->t2, nullptr, BW * n, m2, n, m2, 0);
    if (!(f->tc_on && f->tc_adj &&
          twa::tc_gemm(reinterpret_cast<const float*>(f->t2), BW * n * n, 2 * m2, 2 * m2, f->Ba, n, f->npa, out, n, accumulate,
                  f->d_err, 2.0, st) == 0))
        axis_launch(st, f->t2, nullptr, f->Mi[2], nullptr, out, BW * n * n, m2, n, 1, accumulate);
}

template <int PW_O, int P, bool TRANS, int EP>
void pointwise_o(const float* X, const __nv_bfloat16* W, const float* b, float* Y, float* Z, int B, int cin, int cout,
                 long long K, int acc, cudaStream_t st) {
    const dim3 grid((unsigned)((K + 128 * P - 1) / (128 * P)), (unsigned)((cout + PW_O - 1) / PW_O), (unsigned)(B < 65535 ? B : 65535));
    if (K % 4 == 0 && aligned(X, 16) && aligned(Y, 16) && aligned(Z, 16))
        k_pointwise<PW_O, P, TRANS, EP, true><<<grid, 128, 0, st>>>(X, W, b, Y, Z, B, cin, cout, K, acc);
    else
        k_pointwise<PW_O, P, TRANS, EP, false><<<grid, 128, 0, st>>>(X, W, b, Y, Z, B, cin, cout, K, acc);
}
// Z: where EP_GELU stores gelu(Y), or what EP_GRAD takes gelu' of
template <bool TRANS, int EP>
void pointwise(const float* X, const __nv_bfloat16* W, const float* b, float* Y, float* Z, int B, int cin, int cout,
               long long K, int acc, cudaStream_t st) {
    if (cout <= 4) pointwise_o<4, 4, TRANS, EP>(X, W, b, Y, Z, B, cin, cout, K, acc, st);
    else if (cout <= 8) pointwise_o<8, 4, TRANS, EP>(X, W, b, Y, Z, B, cin, cout, K, acc, st);
    else if (cout <= 16) pointwise_o<16, 4, TRANS, EP>(X, W, b, Y, Z, B, cin, cout, K, acc, st);
    else pointwise_o<32, 2, TRANS, EP>(X, W, b, Y, Z, B, cin, cout, K, acc, st);
}

void pointwise_wgrad(twa_fno* f, const float* dY, const float* X, int B, int cin, int cout, long long K, float* dW,
                     float* db, cudaStream_t st) {
    const dim3 grid(kPwBlocks, (unsigned)(((cout + 31) / 32) * ((cin + 31) / 32)));
    if (K % 4 == 0 && aligned(dY, 16) && aligned(X, 16))
        k_pointwise_wgrad<true><<<grid, 256, WG_SMEM, st>>>(dY, X, B, cin, cout, K, f->part);
    else
        k_pointwise_wgrad<false><<<grid, 256, WG_SMEM, st>>>(dY, X, B, cin, cout, K, f->part);
    k_pointwise_wgrad_sum<<<cout, 128, 0, st>>>(f->part, cin, kPwBlocks, dW, db);
}

}  // namespace

extern "C" {

int twa_fno_create(twa_fno** out, const twa_fno_config* cfg, uint64_t seed) {
    twa_fno* f = nullptr;
    if (!out || !cfg) return ffail(nullptr, TWA_EINVAL, "twa_fno_create: null argument");
    *out = nullptr;
    const twa_fno_config c = *cfg;
    if (c.grid < 4 || c.grid > 128 || c.width < 1 || c.width > 64 || c.modes < 1 || 2 * c.modes > c.grid ||
        c.layers < 1 || c.c_in < 1 || c.c_in > 64 || c.c_out < 1 || c.c_out > 64 ||
        2LL * (2 * c.modes) * (2 * c.modes) * (2 * c.modes) > (long long)c.grid * c.grid * c.grid)
        return ffail(nullptr, TWA_EINVAL,
                     "twa_fno_create: sizes out of range (grid <= 128; width, c_in, c_out <= 64; 2 (2 modes)^3 <= grid^3)");
    f = new twa_fno();
    f->cfg = c;
    const int W = c.width, L = c.layers;
    const long long Mm = kmodes(f);
    long long o = 0;
    f->oP = o; o += (long long)W * c.c_in;
    f->op = o; o += W;
    for (int l = 0; l < L; ++l) {
        f->oR.push_back(o); o += Mm * W * W * 2;
        f->oW.push_back(o); o += (long long)W * W;
        f->ob.push_back(o); o += W;
    }
    f->oQ = o; o += (long long)c.c_out * W;
    f->oq = o; o += c.c_out;
    f->n_params = o;
    auto bail = [&](int rc) {
        twa_fno_destroy(f);
        return rc;
    };
    int rc;
    if ((rc = falloc(f, &f->th, o)) || (rc = falloc(f, &f->th16, o)) || (rc = falloc(f, &f->grad, o)) ||
        (rc = falloc(f, &f->am, o)) || (rc = falloc(f, &f->av, o)))
        return bail(rc);
    const int maxc = (W > c.c_in ? W : c.c_in) > c.c_out ? (W > c.c_in ? W : c.c_in) : c.c_out;
    if ((rc = falloc(f, &f->part, (size_t)maxc * kPwBlocks * (maxc + 1))) ||
        (rc = falloc(f, &f->lpart, (size_t)152 * 64)))
        return bail(rc);
    // truncated unitary DFT matrices (FP64 on the host), kept frequencies {0..m-1} U {n-m..n-1}
    if (fno_prepare() != 0) return bail(ffail(f, TWA_ECUDA, "twa_fno_create: cudaFuncSetAttribute failed"));
    const int n = c.grid, m2 = 2 * c.modes;
    std::vector<float2> mf((size_t)m2 * n), mi((size_t)n * m2);
    for (int i = 0; i < m2; ++i) {
        const int k = (i < c.modes) ? i : n - m2 + i;
        for (int j = 0; j < n; ++j) {
            const double a = -2.0 * M_PI * (double)k * (double)j / (double)n, s = 1.0 / std::sqrt((double)n);
            mf[(size_t)i * n + j] = make_float2((float)(std::cos(a) * s), (float)(std::sin(a) * s));
            mi[(size_t)j * m2 + i] = make_float2((float)(std::cos(a) * s), (float)(-std::sin(a) * s));
        }
    }
    for (int a = 0; a < 3; ++a) {
        if ((rc = falloc(f, &f->Mf[a], mf.size())) || (rc = falloc(f, &f->Mi[a], mi.size()))) return bail(rc);
        cudaMemcpy(f->Mf[a], mf.data(), mf.size() * sizeof(float2), cudaMemcpyHostToDevice);
        cudaMemcpy(f->Mi[a], mi.data(), mi.size() * sizeof(float2), cudaMemcpyHostToDevice);
    }
    // real forms of the x-axis matrices for the tensor-core GEMMs (rows past 2 m2 / n stay zero)
    f->npf = (2 * m2 + 15) / 16 * 16;
    f->npa = (n + 15) / 16 * 16;
    f->tc_fwd = twa::tc_gemm_supported(n, f->npf);
    f->tc_adj = twa::tc_gemm_supported(2 * m2, f->npa);
    if ((rc = falloc(f, &f->d_err, 1))) return bail(rc);
    cudaMemset(f->d_err, 0, sizeof(int));
    if (f->tc_fwd) {
        std::vector<float> bf((size_t)f->npf * n, 0.f);
        for (int i = 0; i < m2; ++i)
            for (int j = 0; j < n; ++j) {
                bf[(size_t)(2 * i) * n + j] = mf[(size_t)i * n + j].x;
                bf[(size_t)(2 * i + 1) * n + j] = mf[(size_t)i * n + j].y;
            }
        if ((rc = falloc(f, &f->Bf, bf.size()))) return bail(rc);
        cudaMemcpy(f->Bf, bf.data(), bf.size() * sizeof(float), cudaMemcpyHostToDevice);
    }
    if (f->tc_adj) {
        std::vector<float> ba((size_t)f->npa * 2 * m2, 0.f);
        for (int j = 0; j < n; ++j)
            for (int i = 0; i < m2; ++i) {
                ba[(size_t)j * 2 * m2 + 2 * i] = mi[(size_t)j * m2 + i].x;
                ba[(size_t)j * 2 * m2 + 2 * i + 1] = -mi[(size_t)j * m2 + i].y;
            }
        if ((rc = falloc(f, &f->Ba, ba.size()))) return bail(rc);
        cudaMemcpy(f->Ba, ba.data(), ba.size() * sizeof(float), cudaMemcpyHostToDevice);
    }
    // initial weights: uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) for pointwise maps, scale 1/(W^2) for R,
    // zero biases, from a fixed linear-congruential stream of the seed (host side)
    // (eight steps of the stream at a time, each lane jumping eight: one step after the other is a chain
    // of multiplications; in pieces of 4 MB, which stay in the host's cache between filling and copying)
    constexpr uint64_t A = 6364136223846793005ULL, Cc = 1442695040888963407ULL;
    uint64_t st = seed * A + Cc;
    std::vector<float> piece((size_t)std::min<long long>(1 << 20, o));
    cudaMemset(f->th, 0, o * sizeof(float));
    auto fill = [&](long long at, long long n, double div) {
        constexpr int LN = 8;
        uint64_t a8 = 1, c8 = 0, x[LN];
        for (int k = 0; k < LN; ++k) {
            c8 = c8 * A + Cc;
            a8 *= A;
            x[k] = st * a8 + c8;   // the k + 1st next value
        }
        const auto value = [div](uint64_t v) { return (float)((((double)(v >> 11) / 9007199254740992.0) * 2.0 - 1.0) / div); };
        for (long long done = 0; done < n;) {
            const long long m = std::min<long long>((long long)piece.size(), n - done);
            float* d = piece.data();
            long long i = 0;
            for (; i + LN <= m; i += LN) {
                st = x[LN - 1];
                for (int k = 0; k < LN; ++k) {
                    d[i + k] = value(x[k]);
                    x[k] = x[k] * a8 + c8;
                }
            }
            for (int k = 0; i < m; ++i, ++k) {   // the last piece only: its size alone is no multiple of eight
                d[i] = value(x[k]);
                st = x[k];
            }
            cudaMemcpy(f->th + at + done, d, (size_t)m * sizeof(float), cudaMemcpyHostToDevice);
            done += m;
        }
    };
    fill(f->oP, (long long)W * c.c_in, std::sqrt((double)c.c_in));
    for (int l = 0; l < L; ++l) {
        fill(f->oR[l], Mm * W * W * 2, (double)W * W);
        fill(f->oW[l], (long long)W * W, std::sqrt((double)W));
    }
    fill(f->oQ, (long long)c.c_out * W, std::sqrt((double)W));
    k_to_bf16<<<blocks_for(o), kThreads>>>(f->th, f->th16, o);
    cudaMemset(f->am, 0, o * sizeof(float));
    cudaMemset(f->av, 0, o * sizeof(float));
    cudaMemset(f->grad, 0, o * sizeof(float));
    if (cudaDeviceSynchronize() != cudaSuccess) {
        cudaGetLastError();
        return bail(ffail(f, TWA_ECUDA, "twa_fno_create: setup failed"));
    }
    *out = f;
    return TWA_OK;
}

int twa_fno_destroy(twa_fno* f) {
    if (!f) return TWA_OK;
    for (void* p : f->acts) cudaFree(p);
    for (void* p : f->allocs) cudaFree(p);
    delete f;
    return TWA_OK;
}

long long twa_fno_num_params(const twa_fno* f) { return f ? f->n_params : 0; }

int twa_fno_set_params(twa_fno* f, const float* src, void* stream) {
    if (!f || !src) return ffail(f, TWA_EINVAL, "twa_fno_set_params: null argument");
    cudaStream_t st = (cudaStream_t)stream;
    FC(cudaMemcpyAsync(f->th, src, f->n_params * sizeof(float), cudaMemcpyDeviceToDevice, st));
    k_to_bf16<<<blocks_for(f->n_params), kThreads, 0, st>>>(f->th, f->th16, f->n_params);
    FC(cudaMemsetAsync(f->am, 0, f->n_params * sizeof(float), st));
    FC(cudaMemsetAsync(f->av, 0, f->n_params * sizeof(float), st));
    f->step = 0;
    FC(cudaGetLastError());
    return TWA_OK;
}

int twa_fno_get_params(twa_fno* f, float* dst, int which, void* stream) {
    if (!f || !dst) return ffail(f, TWA_EINVAL, "twa_fno_get_params: null argument");
    const float* src = which == 1 ? f->grad : f->th;
    FC(cudaMemcpyAsync(dst, src, f->n_params * sizeof(float), cudaMemcpyDeviceToDevice, (cudaStream_t)stream));
    return TWA_OK;
}

int twa_fno_forward(twa_fno* f, const float* x, int B, float* y, void* stream) {
    if (!f || !x || !y || B < 1) return ffail(f, TWA_EINVAL, "twa_fno_forward: bad argument");
    cudaStream_t st = (cudaStream_t)stream;
    if (int rc = ensure_batch(f, B)) return rc;
    const int W = f->cfg.width, L = f->cfg.layers;
    const long long K = kcells(f), Mm = kmodes(f), BW = (long long)B * W;
    const __nv_bfloat16* P = f->th16;
    pointwise<false, EP_NONE>(x, P + f->oP, f->th + f->op, f->h[0], nullptr, B, f->cfg.c_in, W, K, 0, st);
    for (int l = 0; l < L; ++l) {
        dft_fwd(f, f->h[l], f->s[l], BW, st);
        mix_launch<false>(f->s[l], P + f->oR[l], f->mixed, B, W, Mm, st);
        dft_adj(f, f->mixed, f->z[l], BW, 0, st);
        if (l < L - 1)
            pointwise<false, EP_GELU>(f->h[l], P + f->oW[l], f->th + f->ob[l], f->z[l], f->h[l + 1], B, W, W, K, 1, st);
        else
            pointwise<false, EP_NONE>(f->h[l], P + f->oW[l], f->th + f->ob[l], f->z[l], nullptr, B, W, W, K, 1, st);
    }
    pointwise<false, EP_NONE>(f->h[L], P + f->oQ, f->th + f->oq, y, nullptr, B, W, f->cfg.c_out, K, 0, st);
    f->x_in = x;
    f->last_b = B;
    FC(cudaGetLastError());
    return TWA_OK;
}

int twa_fno_backward(twa_fno* f, const float* dy, int B, float* dx, void* stream) {
    if (!f || !dy || B != f->last_b || !f->x_in) return ffail(f, TWA_EINVAL, "twa_fno_backward: call after twa_fno_forward with the same batch");
    cudaStream_t st = (cudaStream_t)stream;
    const int W = f->cfg.width, L = f->cfg.layers;
    const long long K = kcells(f), Mm = kmodes(f), BW = (long long)B * W;
    const __nv_bfloat16* P = f->th16;
    float* g = f->grad;
    pointwise_wgrad(f, dy, f->h[L], B, W, f->cfg.c_out, K, g + f->oQ, g + f->oq, st);
    pointwise<true, EP_NONE>(dy, P + f->oQ, nullptr, f->dz, nullptr, B, f->cfg.c_out, W, K, 0, st);
    for (int l = L - 1; l >= 0; --l) {
        pointwise_wgrad(f, f->dz, f->h[l], B, W, W, K, g + f->oW[l], g + f->ob[l], st);
        // spectral branch: dmixed = A dz, dR += dmixed conj(s), ds = R^H dmixed (in t2, which the adjoint
        // transform reads before it writes it), dh = Re A^H ds
        float2* ds = f->t2;
        dft_fwd(f, f->dz, f->mixed, BW, st);
        mix_wgrad_launch(f->mixed, f->s[l], g + f->oR[l], B, W, Mm, st);
        mix_launch<true>(f->mixed, P + f->oR[l], ds, B, W, Mm, st);
        dft_adj(f, ds, f->dz2, BW, 0, st);
        // dh += W^T dz, and for the layer below dz = dh gelu'(z)
        if (l > 0)
            pointwise<true, EP_GRAD>(f->dz, P + f->oW[l], nullptr, f->dz2, f->z[l - 1], B, W, W, K, 1, st);
        else
            pointwise<true, EP_NONE>(f->dz, P + f->oW[l], nullptr, f->dz2, nullptr, B, W, W, K, 1, st);
        std::swap(f->dz, f->dz2);
    }
    pointwise_wgrad(f, f->dz, f->x_in, B, f->cfg.c_in, W, K, g + f->oP, g + f->op, st);
    if (dx) pointwise<true, EP_NONE>(f->dz, P + f->oP, nullptr, dx, nullptr, B, W, f->cfg.c_in, K, 0, st);
    FC(cudaGetLastError());
    return TWA_OK;
}

int twa_fno_zero_grad(twa_fno* f, void* stream) {
    if (!f) return ffail(nullptr, TWA_EINVAL, "null model");
    FC(cudaMemsetAsync(f->grad, 0, f->n_params * sizeof(float), (cudaStream_t)stream));
    return TWA_OK;
}

int twa_fno_adamw(twa_fno* f, float lr, float beta1, float beta2, float eps, float weight_decay, void* stream) {
    if (!f) return ffail(nullptr, TWA_EINVAL, "null model");
    f->step += 1;
    const float c1 = 1.f - (float)std::pow((double)beta1, (double)f->step);
    const float c2 = 1.f - (float)std::pow((double)beta2, (double)f->step);
    k_adamw<<<blocks_for(f->n_params), kThreads, 0, (cudaStream_t)stream>>>(f->th, f->grad, f->am, f->av, f->th16,
                                                                          f->n_params, lr, beta1, beta2, eps,
                                                                          weight_decay, c1, c2);
    FC(cudaGetLastError());
    return TWA_OK;
}

int twa_fno_mse(twa_fno* f, const float* y, const float* t, long long n, float* loss, float* dy, void* stream) {
    if (!f || !y || !t || !loss || n < 1) return ffail(f, TWA_EINVAL, "twa_fno_mse: bad argument");
    cudaStream_t st = (cudaStream_t)stream;
    const int nb = 152 * 4;
    k_mse_part<<<nb, 256, 0, st>>>(y, t, n, dy, f->lpart);
    k_mse_final<<<1, 256, 0, st>>>(f->lpart, nb, n, loss);
    FC(cudaGetLastError());
    return TWA_OK;
}

const char* twa_fno_last_error(const twa_fno* f) { return f ? f->err.c_str() : ""; }

int twa_fno_set_tensor_cores(twa_fno* f, int on) {
    if (!f) return ffail(nullptr, TWA_EINVAL, "twa_fno_set_tensor_cores: null handle");
    f->tc_on = on != 0;
    return TWA_OK;
}

int twa_fno_tensor_core_shapes(const twa_fno* f) {
    if (!f) return 0;
    return (f->tc_fwd ? 1 : 0) | (f->tc_adj ? 2 : 0);
}

int twa_fno_sync_status(twa_fno* f, void* stream) {
    if (!f) return ffail(nullptr, TWA_EINVAL, "twa_fno_sync_status: null handle");
    FC(cudaStreamSynchronize((cudaStream_t)stream));
    int w = 0;
    FC(cudaMemcpy(&w, f->d_err, sizeof(int), cudaMemcpyDeviceToHost));
    FC(cudaMemset(f->d_err, 0, sizeof(int)));
    if (w & twa::TC_ERR_TIMEOUT_BIT) return ffail(f, TWA_ETIMEOUT, "a tensor-core GEMM wait gave up");
    return TWA_OK;
}

int twa_tc_gemm(const float* A, long long P, long long K, long long lda, const float* Bt, int N, int Np, float* C,
                long long ldc, int accumulate, int* err, void* stream) {
    if (!A || !Bt || !C || !err || P <= 0 || N <= 0 || N > Np || lda < K || ldc < N)
        return ffail(nullptr, TWA_EINVAL, "twa_tc_gemm: bad argument");
    const int rc = twa::tc_gemm(A, P, K, lda, Bt, N, Np, C, ldc, accumulate, err, 2.0, (cudaStream_t)stream);
    if (rc == -1)
        return ffail(nullptr, TWA_EINVAL,
                     "twa_tc_gemm: unsupported shape or alignment (K a multiple of 32 up to 128, Np a multiple of 16 "
                     "in [16, 256], 16-byte aligned A and Bt, lda * 4 a multiple of 16)");
    if (rc) return ffail(nullptr, TWA_ECUDA, "twa_tc_gemm: tensor map or launch failed");
    return TWA_OK;
}

}  // extern "C"

namespace {
// Features of one TWA snapshot on the mode grid (FFT index order), with nu = n_tot / grid^3 the mean
// occupation per mode:
//   x0 = log10(1 + n_cl) / 8,  x1 = (n_est - n_cl) / (n_cl + nu),  x2 = log10(n_tot) - 9,
//   x3 = |m| / (grid / 2);   target t = (n_ref - n_cl) / (n_cl + nu)  (the correction spectrum relative
// to the occupation, floored at the mean occupation).
__global__ void k_features(const double* __restrict__ ncl, const double* __restrict__ nest, const double* __restrict__ nref,
                           double lg_ntot, double nu, int n, float* __restrict__ x, float* __restrict__ t) {
    const long long K = (long long)n * n * n;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < K; k += (long long)gridDim.x * blockDim.x) {
        const double c = ncl[k];
        const double sc = 1.0 / ((c > 0.0 ? c : 0.0) + nu);
        const int ix = (int)(k % n), iy = (int)((k / n) % n), iz = (int)(k / ((long long)n * n));
        const double mx = ix < n / 2 ? ix : ix - n, my = iy < n / 2 ? iy : iy - n, mz = iz < n / 2 ? iz : iz - n;
        x[k] = (float)(log10(1.0 + (c > 0.0 ? c : 0.0)) / 8.0);
        x[K + k] = (float)((nest[k] - c) * sc);
        x[2 * K + k] = (float)(lg_ntot - 9.0);
        x[3 * K + k] = (float)(sqrt(mx * mx + my * my + mz * mz) / (0.5 * n));
        if (t) t[k] = (float)((nref[k] - c) * sc);
    }
}
}  // namespace

extern "C" int twa_fno_features(const double* nk_cl, const double* nk_est, const double* nk_ref, double n_tot, int grid,
                                float* x, float* t, void* stream) {
    if (!nk_cl || !nk_est || !x || grid < 2 || (t && !nk_ref) || !(n_tot > 0)) {
        twa_set_global_error("twa_fno_features: bad argument");
        return TWA_EINVAL;
    }
    const long long K = (long long)grid * grid * grid;
    k_features<<<blocks_for(K), kThreads, 0, (cudaStream_t)stream>>>(nk_cl, nk_est, nk_ref, std::log10(n_tot),
                                                                    n_tot / (double)K, grid, x, t);
    if (cudaGetLastError() != cudaSuccess) {
        twa_set_global_error("twa_fno_features: launch failed");
        return TWA_ECUDA;
    }
    return TWA_OK;
}

extern "C" {

}  // extern "C"
