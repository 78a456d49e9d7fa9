// fch_fno.cu -- a Fourier neural operator (FNO) that predicts the initial iterate
// of the PSD iteration (Sec. 3.3 leaves v_0 free): forward pass, backward pass,
// mean-square loss and Adam, all in FP32 on this library's own kernels and its
// own batched real 2D transforms (no cuFFT, no cuBLAS).
//
// Network (restating Li et al.'s Fourier neural operator): two input channels per
// point, a = (u^n, (u* - u^n)/s), u* the extrapolation of eq. (Richardson), s the
// RMS of u* - u^n; output y = predicted (u^{n+1} - u*)/s.
//   h_0 = P a + bP;  h_{l+1} = act_l(W_l h_l + b_l + S_l(h_l));  y = Q2 GELU(Q1 h_L + bQ1) + bQ2
//   S(h)[o] = C2R(H(sum_i R[m][o][i] R2C(h[i])(m)))  over the retained modes m,
// act = GELU (x Phi(x), with erf) except after the last layer (identity). Retained
// modes: kx in [0, M), ky in {0..M-1} and {N-M+1..N-1}, weight index
// kx (2M-1) + kyi with ky = kyi (kyi < M) or -(kyi - M + 1). H replaces the kx = 0
// column of the retained modes by its Hermitian part (Y(ky) + conj Y(-ky))/2, the
// part a real inverse transform reads. The backward pass uses the adjoints: of C2R
// on retained modes w(kx)/N^2 R2C (w = 1 at kx = 0, else 2), of R2C
// N^2 C2R(v(kx) .), v = 1 at kx = 0, else 1/2, both through H at kx = 0.
//
// Layouts: fields [b][c][y][x] (channel fields contiguous, n x n each); spectra as
// the library's transforms write them, kx-major [field][kx][ky]; parameters one
// flat float vector in the order P, bP, {W_l, b_l, R_l} for each layer, Q1, bQ1,
// Q2, bQ2, with R_l as [K][W_out][W_in] complex (re, im interleaved).
// Weight gradients are summed over points in a fixed order (per-block partials,
// then one pass over the blocks), so a backward pass is deterministic.
#include <cuda.h> // CUtensorMap and its enums (the encoder is fetched at run time)
#include <cuda_bf16.h>
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include "../../include/fch.h"
#include "fch_fnomodes.cuh"
#include "fch_internal.h"
#include "fch_tc.cuh"
#include "fch_tmap.h"

namespace {

constexpr int kMaxW2 = 128;  // hidden channels of the projection
constexpr int kMaxQ1 = 2048; // its first layer's weights, W2 W

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float x)
{
    return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// Two floats in one 64-bit register, for the packed FP32 instructions of this GPU
// (add / mul / fma .rn.f32x2: both lanes in one instruction).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 x2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 x2_split(f32x2 v)
{
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return make_float2(a, b);
}
__device__ __forceinline__ f32x2 x2_fma(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 x2_mul(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 x2_add(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// GELU of two values at once for the tensor-core inference kernels. erf comes from the
// rational approximation of Abramowitz and Stegun, Handbook of Mathematical Functions,
// eq. 7.1.28: for u >= 0, 1 - erf(u) = p(u)^-16 with p(u) = 1 + a1 u + ... + a6 u^6,
// |error| <= 3e-7. With h = x/2 and a = |h| (u = a sqrt 2),
//   GELU(x) = x/2 (1 + erf(x / sqrt 2)) = (a + h) - a p(u)^-16,
// which for x < 0 is -a p^-16 itself (no cancellation); a is capped in the last term. One reciprocal per value (with
// a Newton step), the rest packed: about twelve instructions a value against the
// library erff's branches. In float, p^-16 carries ~2e-6 relative rounding: GELU
// within 0.5 |x| 3e-6. Its outputs feed bfloat16 operands (relative rounding 2^-9) or
// FP32 sums with bfloat16 weights.
__device__ __forceinline__ f32x2 gelu_as2(f32x2 x)
{
    const f32x2 h = x2_mul(x, x2(0.5f, 0.5f));
    const f32x2 a = h & 0x7FFFFFFF7FFFFFFFull; // |h|
    // the tail term takes |h| capped at 5.65 (u = |h| sqrt 2 at most 8, where 1 - erf is
    // 1e-29 and p stays finite for the Newton step)
    const float2 as = x2_split(a);
    const f32x2 acn = x2(-fminf(as.x, 5.65f), -fminf(as.y, 5.65f));
    const f32x2 u = x2_mul(acn, x2(-1.41421356237309505f, -1.41421356237309505f));
    f32x2 p = x2_fma(x2(0.0000430638f, 0.0000430638f), u, x2(0.0002765672f, 0.0002765672f));
    p = x2_fma(p, u, x2(0.0001520143f, 0.0001520143f));
    p = x2_fma(p, u, x2(0.0092705272f, 0.0092705272f));
    p = x2_fma(p, u, x2(0.0422820123f, 0.0422820123f));
    p = x2_fma(p, u, x2(0.0705230784f, 0.0705230784f));
    p = x2_fma(p, u, x2(1.0f, 1.0f)); // in [1, 22]
    const float2 ps = x2_split(p);
    f32x2 r = x2(rcp_approx(ps.x), rcp_approx(ps.y));
    r = x2_fma(r, x2_fma(p ^ 0x8000000080000000ull, r, x2(1.0f, 1.0f)), r); // Newton: r (2 - p r)
    r = x2_mul(r, r);
    r = x2_mul(r, r);
    r = x2_mul(r, r);
    r = x2_mul(r, r); // p^-16
    return x2_fma(acn, r, x2_add(a, h));
}

// ky of retained-mode row kyi
__device__ __forceinline__ int mode_ky(int kyi, int M, int n) { return kyi < M ? kyi : n - (kyi - M + 1); }

// a weight as float: the forward pass reads FP32 weights, or (inference with
// fch_fno_set_bf16) their bfloat16 copy; sums stay in FP32 either way
__device__ __forceinline__ float wld(const float *p, long i) { return p[i]; }
__device__ __forceinline__ float wld(const __nv_bfloat16 *p, long i) { return __bfloat162float(p[i]); }
__device__ __forceinline__ float2 wld2(const float *p, long i) { return make_float2(p[2 * i], p[2 * i + 1]); }
__device__ __forceinline__ float2 wld2(const __nv_bfloat16 *p, long i)
{
    return __bfloat1622float2(reinterpret_cast<const __nv_bfloat162 *>(p)[i]);
}

__global__ void fno_to_bf16(const float *__restrict__ w, __nv_bfloat16 *__restrict__ out, long cnt)
{
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < cnt) out[t] = __float2bfloat16_rn(w[t]);
}

// h0[b][c][p] = sum_i P[c][i] a[b][i][p] + bP[c]: the channel counts fixed at compile time,
// loops unrolled, each output channel one multiply-add chain and one store at a running
// pointer (bf16 output: the tensor-core pass, whose kernels read h rounded to bf16)
__device__ __forceinline__ void put(float *p, float v) { *p = v; }
__device__ __forceinline__ void put(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }
template <typename WT, int W, int CIN, typename HT = float>
__global__ void __launch_bounds__(256) fno_lift_t(const float *__restrict__ a, const WT *__restrict__ P,
                                                  const WT *__restrict__ bP, HT *__restrict__ h, long pts, int n2)
{
    __shared__ float ps[W * CIN], bs[W];
    for (int i = threadIdx.x; i < W * CIN; i += blockDim.x) ps[i] = wld(P, i);
    for (int i = threadIdx.x; i < W; i += blockDim.x) bs[i] = wld(bP, i);
    __syncthreads();
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= pts) return;
    const long b = t / n2, p = t - b * n2;
    float in[CIN];
#pragma unroll
    for (int i = 0; i < CIN; i++) in[i] = __ldcs(a + (b * CIN + i) * n2 + p);
    HT *hp = h + b * W * n2 + p;
#pragma unroll
    for (int c = 0; c < W; c++) {
        float acc = bs[c];
#pragma unroll
        for (int i = 0; i < CIN; i++) acc = fmaf(ps[c * CIN + i], in[i], acc);
        put(hp, acc);
        hp += n2;
    }
}

// z[b][c][p] = sum_j Wl[c][j] h[b][j][p] + bl[c] + s[b][c][p];  out = act(z)
// (W, the channel count, is a compile-time constant so the per-point channel vectors stay
// in registers). A thread takes two neighbouring points: each 16-byte read of four weights
// from shared memory feeds eight multiply-adds, where one point and scalar reads made the
// kernel wait on shared memory (one read a multiply-add; 128^2, batch 8, W = 32: 26 us for
// 67 MB).
template <int W, typename WT = float>
__global__ void __launch_bounds__(128) fno_pointwise(const float *__restrict__ h, const float *__restrict__ s,
                                                     const WT *__restrict__ Wl, const WT *__restrict__ bl,
                                                     float *__restrict__ z, float *__restrict__ out, int B, int n2,
                                                     int act)
{
    __shared__ __align__(16) float ws[W * W];
    __shared__ float bs[W];
    for (int i = threadIdx.x; i < W * W; i += blockDim.x) ws[i] = wld(Wl, i);
    for (int i = threadIdx.x; i < W; i += blockDim.x) bs[i] = wld(bl, i);
    __syncthreads();
    const long t = 2 * ((long)blockIdx.x * blockDim.x + threadIdx.x);
    if (t >= (long)B * n2) return;
    const int b = (int)(t / n2), p = (int)(t - (long)b * n2);
    const long o0 = (long)b * W * n2 + p;
    float2 in[W];
#pragma unroll
    for (int j = 0; j < W; j++) in[j] = *(const float2 *)(h + o0 + (long)j * n2);
#pragma unroll 2
    for (int c = 0; c < W; c++) {
        const long o = o0 + (long)c * n2;
        const float2 sv = *(const float2 *)(s + o);
        float2 acc = make_float2(bs[c] + sv.x, bs[c] + sv.y);
#pragma unroll
        for (int j = 0; j < W; j += 4) {
            const float4 w = *(const float4 *)(ws + c * W + j);
            acc.x = fmaf(w.x, in[j].x, acc.x);
            acc.y = fmaf(w.x, in[j].y, acc.y);
            acc.x = fmaf(w.y, in[j + 1].x, acc.x);
            acc.y = fmaf(w.y, in[j + 1].y, acc.y);
            acc.x = fmaf(w.z, in[j + 2].x, acc.x);
            acc.y = fmaf(w.z, in[j + 2].y, acc.y);
            acc.x = fmaf(w.w, in[j + 3].x, acc.x);
            acc.y = fmaf(w.w, in[j + 3].y, acc.y);
        }
        *(float2 *)(z + o) = acc;
        *(float2 *)(out + o) = act ? make_float2(gelu(acc.x), gelu(acc.y)) : acc;
    }
}

// y[b][p] = bQ2 + sum_d Q2[d] GELU(bQ1[d] + sum_c Q1[d][c] h[b][c][p]); two points a thread
// and the weights in shared memory, as fno_pointwise (read from global memory one weight a
// multiply-add it took 65 us for 131072 points, W = 32, W2 = 64)
template <int W, typename WT = float>
__global__ void __launch_bounds__(128) fno_project(const float *__restrict__ h, const WT *__restrict__ Q1,
                                                   const WT *__restrict__ bQ1, const WT *__restrict__ Q2,
                                                   const WT *__restrict__ bQ2, float *__restrict__ y, int B, int n2,
                                                   int W2)
{
    __shared__ __align__(16) float ws[kMaxQ1];
    __shared__ float bs[kMaxW2], qs[kMaxW2];
    for (int i = threadIdx.x; i < W2 * W; i += blockDim.x) ws[i] = wld(Q1, i);
    for (int i = threadIdx.x; i < W2; i += blockDim.x) {
        bs[i] = wld(bQ1, i);
        qs[i] = wld(Q2, i);
    }
    __syncthreads();
    const long t = 2 * ((long)blockIdx.x * blockDim.x + threadIdx.x);
    if (t >= (long)B * n2) return;
    const int b = (int)(t / n2), p = (int)(t - (long)b * n2);
    float2 in[W];
#pragma unroll
    for (int c = 0; c < W; c++) in[c] = *(const float2 *)(h + ((long)b * W + c) * n2 + p);
    const float b2 = wld(bQ2, 0);
    float2 acc = make_float2(b2, b2);
    for (int d = 0; d < W2; d++) {
        float2 zq = make_float2(bs[d], bs[d]);
#pragma unroll
        for (int c = 0; c < W; c += 4) {
            const float4 w = *(const float4 *)(ws + d * W + c);
            zq.x = fmaf(w.x, in[c].x, zq.x);
            zq.y = fmaf(w.x, in[c].y, zq.y);
            zq.x = fmaf(w.y, in[c + 1].x, zq.x);
            zq.y = fmaf(w.y, in[c + 1].y, zq.y);
            zq.x = fmaf(w.z, in[c + 2].x, zq.x);
            zq.y = fmaf(w.z, in[c + 2].y, zq.y);
            zq.x = fmaf(w.w, in[c + 3].x, zq.x);
            zq.y = fmaf(w.w, in[c + 3].y, zq.y);
        }
        acc.x = fmaf(qs[d], gelu(zq.x), acc.x);
        acc.y = fmaf(qs[d], gelu(zq.y), acc.y);
    }
    y[t] = acc.x;
    y[t + 1] = acc.y;
}

// Backward of the projection and the loss mean((y - target)^2): per point dy, the
// hidden activations q, their gradients dzq and dh = Q1^T dzq; also (y - target)^2
// per point for the loss.
template <int W>
__global__ void fno_project_bwd(const float *__restrict__ h, const float *__restrict__ Q1,
                                const float *__restrict__ bQ1, const float *__restrict__ Q2,
                                const float *__restrict__ y, const float *__restrict__ target, float *__restrict__ dy,
                                float *__restrict__ q, float *__restrict__ dzq, float *__restrict__ dh,
                                float *__restrict__ sq, int B, int n2, int W2, float scale)
{
    __shared__ __align__(16) float ws[kMaxQ1];
    __shared__ float bs[kMaxW2], qs[kMaxW2];
    for (int i = threadIdx.x; i < W2 * W; i += blockDim.x) ws[i] = Q1[i];
    for (int i = threadIdx.x; i < W2; i += blockDim.x) {
        bs[i] = bQ1[i];
        qs[i] = Q2[i];
    }
    __syncthreads();
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)B * n2) return;
    const int b = (int)(t / n2), p = (int)(t - (long)b * n2);
    float in[W], g[W];
#pragma unroll
    for (int c = 0; c < W; c++) {
        in[c] = h[((long)b * W + c) * n2 + p];
        g[c] = 0.f;
    }
    const float r = y[t] - target[t];
    const float d = scale * r;
    dy[t] = d;
    sq[t] = r * r;
    for (int k = 0; k < W2; k++) {
        float4 w[W / 4];
        float zq = bs[k];
#pragma unroll
        for (int c = 0; c < W; c += 4) {
            w[c / 4] = *(const float4 *)(ws + k * W + c);
            zq = fmaf(w[c / 4].x, in[c], zq);
            zq = fmaf(w[c / 4].y, in[c + 1], zq);
            zq = fmaf(w[c / 4].z, in[c + 2], zq);
            zq = fmaf(w[c / 4].w, in[c + 3], zq);
        }
        const long o = ((long)b * W2 + k) * n2 + p;
        q[o] = gelu(zq);
        const float dz = d * qs[k] * gelu_grad(zq);
        dzq[o] = dz;
#pragma unroll
        for (int c = 0; c < W; c += 4) {
            g[c] = fmaf(w[c / 4].x, dz, g[c]);
            g[c + 1] = fmaf(w[c / 4].y, dz, g[c + 1]);
            g[c + 2] = fmaf(w[c / 4].z, dz, g[c + 2]);
            g[c + 3] = fmaf(w[c / 4].w, dz, g[c + 3]);
        }
    }
#pragma unroll
    for (int c = 0; c < W; c++) dh[((long)b * W + c) * n2 + p] = g[c];
}

// Backward of a Fourier layer's pointwise part: dz = dout act'(z); dh = Wl^T dz.
template <int W>
__global__ void fno_pointwise_bwd(const float *__restrict__ dout, const float *__restrict__ z,
                                  const float *__restrict__ Wl, float *__restrict__ dz, float *__restrict__ dh,
                                  int B, int n2, int act)
{
    __shared__ __align__(16) float ws[W * W];
    for (int i = threadIdx.x; i < W * W; i += blockDim.x) ws[i] = Wl[i];
    __syncthreads();
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)B * n2) return;
    const int b = (int)(t / n2), p = (int)(t - (long)b * n2);
    float g[W], acc[W];
#pragma unroll
    for (int c = 0; c < W; c++) {
        const long o = ((long)b * W + c) * n2 + p;
        g[c] = act ? dout[o] * gelu_grad(z[o]) : dout[o];
        dz[o] = g[c];
        acc[c] = 0.f;
    }
#pragma unroll
    for (int c = 0; c < W; c++)
#pragma unroll
        for (int j = 0; j < W; j++) acc[j] += ws[c * W + j] * g[c];
#pragma unroll
    for (int j = 0; j < W; j++) dh[((long)b * W + j) * n2 + p] = acc[j];
}

// Y[b W + o](m) = sum_i R[m][o][i] X[b W + i](m) on the retained modes, written
// through H at kx = 0 (work item: one mode, or at kx = 0 the pair ky, -ky).
// X and Y are spectra [field][kx][ky]; S = (n/2 + 1) n complex per field.
template <typename WT>
__global__ void fno_mix(const float2 *__restrict__ X, const WT *__restrict__ R, float2 *__restrict__ Y,
                        int B, int W, int M, int n)
{
    const int items = M + (M - 1) * (2 * M - 1);
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)B * W * items) return;
    const int it = (int)(t % items), o = (int)((t / items) % W), b = (int)(t / ((long)items * W));
    const long S = (long)(n / 2 + 1) * n;
    const int K2 = 2 * M - 1;
    auto mixed = [&](int kx, int kyi) {
        const int ky = mode_ky(kyi, M, n);
        const long r = ((long)(kx * K2 + kyi) * W + o) * W; // complex index of R[m][o][0]
        float re = 0.f, im = 0.f;
        for (int i = 0; i < W; i++) {
            const float2 x = X[((long)b * W + i) * S + (long)kx * n + ky];
            const float2 w = wld2(R, r + i);
            re += w.x * x.x - w.y * x.y;
            im += w.x * x.y + w.y * x.x;
        }
        return make_float2(re, im);
    };
    float2 *Yf = Y + ((long)b * W + o) * S;
    if (it < M) { // kx = 0: ky = it and -it
        const int ky = it;
        const float2 yp = mixed(0, ky);
        if (ky == 0) {
            Yf[0] = make_float2(yp.x, 0.f);
        } else {
            const float2 ym = mixed(0, ky + M - 1);
            const float2 hh = make_float2(0.5f * (yp.x + ym.x), 0.5f * (yp.y - ym.y));
            Yf[ky] = hh;
            Yf[n - ky] = make_float2(hh.x, -hh.y);
        }
    } else {
        const int j = it - M, kx = 1 + j / K2, kyi = j % K2;
        Yf[(long)kx * n + mode_ky(kyi, M, n)] = mixed(kx, kyi);
    }
}

// ---------------------------------------------------------------------------
// Inference with the spectral convolutions as truncated DFTs over the retained
// modes (fch_fno_set_bf16(f, 2)): for a layer input h[b][i][y][x],
//   X[b][i][y][kx] = sum_x h (cos - i sin)(2 pi kx x / n),  kx < M     (rows)
//   Y[b][i][kyi][kx] = sum_y X e^{-2 pi i ky y / n}                     (columns)
//   Z[b][o][kyi][kx] = sum_i R[m][o][i] Y[b][i][kyi][kx], m = kx (2M-1) + kyi
//   V[b][o][y][kx] = sum_kyi Z e^{+2 pi i ky y / n}
//   S[b][o][y][x] = (1/n^2) sum_kx w(kx) Re(V e^{+2 pi i kx x / n}),  w(0) = 1, else 2
// which is the C2R of the retained spectrum through H (the real part of the kx = 0
// sum is what H keeps), without the full 2D transforms of every channel. The row
// DFT, a GEMM with K = n, runs on the tensor cores (tcgen05, BF16 operands, FP32
// sums); the other stages are small and run as plain kernels in FP32.

constexpr int kTcRows = 128, kTcLBO = 144, kTcSBO = 8 * kTcLBO, kTcNB = 32;
constexpr uint64_t kTcBound = 1000000000ull; // ns an mbarrier wait lasts before a kernel gives up

// Bt[j][x] (bf16): cos(2 pi j x / n) for j < 16, -sin(2 pi (j - 16) x / n) for j >= 16;
// tw[kx][x] (float2): (cos, sin)(2 pi kx x / n), kx < 16; At[j][x] (may be null): tw rounded
// to bf16, cos for j < 16, sin for j >= 16
__global__ void fno_dft_tables(__nv_bfloat16 *__restrict__ Bt, float2 *__restrict__ tw,
                               __nv_bfloat16 *__restrict__ At, int n)
{
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 16L * n) return;
    const int kx = (int)(t / n), x = (int)(t - (long)kx * n);
    double sn, cs;
    sincospi(2.0 * (double)((kx * (long)x) % n) / (double)n, &sn, &cs);
    Bt[(long)kx * n + x] = __double2bfloat16(cs);
    Bt[(long)(16 + kx) * n + x] = __double2bfloat16(-sn);
    tw[(long)kx * n + x] = make_float2((float)cs, (float)sn);
    if (At) {
        At[(long)kx * n + x] = __float2bfloat16_rn((float)cs);
        At[(long)(16 + kx) * n + x] = __float2bfloat16_rn((float)sn);
    }
}

// X[r][kx] = (D[r][kx], D[r][16 + kx]) with D = h Bt^T over K = n, h the bf16 activations:
// one CTA of 128 threads per 128 rows, K in chunks of 64 (128 bytes a row). A chunk of the
// rows and of the table arrive as tiles of two tensor maps with the 128-byte swizzle, the
// layout the tensor core reads, kDftStages chunks ahead; thread 0 alone starts the copies
// and issues four K = 16 MMAs a chunk into a 128 x 32 FP32 accumulator in tensor memory; a
// chunk's `full` mbarrier counts its bytes, its `mma` mbarrier the MMAs that free the
// stage. Rows past R read as zero. A wait that runs out of time (1 s) sets *err; the CTA
// then stops, waits (bounded) for the copies and MMAs it issued, frees its tensor memory
// and returns.
// Bound by reading h. With h in FP32 every CTA's threads rounded each chunk through shared
// memory: 134 MB at 1024^2, 32 channels, 38.5 us; the values are the same, rounded once by
// the kernel that writes them.
constexpr int kDftKc = 64;                                  // K of a chunk (four K = 16 MMAs)
constexpr int kDftStages = 4;
constexpr int kDftABytes = kTcRows * kDftKc * 2, kDftBBytes = kTcNB * kDftKc * 2; // 16 KB, 4 KB
// the stages, then the mbarriers and the tensor-memory address, and 1 KB of slack to
// align the tiles to 1024 bytes
constexpr int kRowdftSmem = kDftStages * (kDftABytes + kDftBBytes) + 128 + 1024;

__global__ void __launch_bounds__(128) fno_rowdft_tc(const __grid_constant__ CUtensorMap amap,
                                                     const __grid_constant__ CUtensorMap bmap,
                                                     float2 *__restrict__ X, int R, int n, int *err)
{
    extern __shared__ unsigned char dsm_raw[];
    // swizzled tiles want 1024-byte alignment: the window's start rounded up
    unsigned char *sA = dsm_raw + ((1024u - (fch::tc::smem_u32(dsm_raw) & 1023u)) & 1023u);
    unsigned char *sB = sA + kDftStages * kDftABytes;
    uint64_t *full = reinterpret_cast<uint64_t *>(sB + kDftStages * kDftBBytes), *mmab = full + kDftStages;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(mmab + kDftStages);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long row0 = (long)blockIdx.x * kTcRows;
    const int nch = n / kDftKc;
    if (warp == 0) {
        fch::tc::tmem_alloc(tslot, 32);
        fch::tc::tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < kDftStages; i++) {
            fch::tc::mbar_init(&full[i], 1);
            fch::tc::mbar_init(&mmab[i], 1);
        }
        fch::tc::mbar_init_fence();
    }
    fch::tc::fence_before_sync();
    __syncthreads();
    fch::tc::fence_after_sync();
    const uint32_t tmem = *tslot;
    bool ok = true;
    if (tid == 0) {
        auto fetch = [&](int c) {
            const int st = c % kDftStages;
            fch::tc::mbar_expect_tx(&full[st], kDftABytes + kDftBBytes);
            fch::tc::tma_load_2d(sA + st * kDftABytes, &amap, c * kDftKc, (int)row0, &full[st]);
            fch::tc::tma_load_2d(sB + st * kDftBBytes, &bmap, c * kDftKc, 0, &full[st]);
        };
        constexpr uint32_t idesc = fch::tc::idesc_bf16_f32(kTcRows, kTcNB);
        int fetched = nch < kDftStages ? nch : kDftStages, issued = 0;
        for (int c = 0; c < fetched; c++) fetch(c);
        for (int c = 0; c < nch && ok; c++) {
            const int st = c % kDftStages;
            ok = fch::tc::mbar_wait(&full[st], (uint32_t)((c / kDftStages) & 1), kTcBound);
            if (!ok) break;
            const uint32_t sa = fch::tc::smem_u32(sA + st * kDftABytes), sb = fch::tc::smem_u32(sB + st * kDftBBytes);
#pragma unroll
            for (int k = 0; k < kDftKc / 16; k++)
                fch::tc::mma_bf16(tmem, fch::tc::smem_desc_sw128(sa + 32 * k), fch::tc::smem_desc_sw128(sb + 32 * k),
                                  idesc, (c | k) != 0);
            fch::tc::mma_commit(&mmab[st]);
            issued = c + 1;
            // the stage of the chunk before is free once its MMAs are done: refill it
            const int pc = c - 1, nc = pc + kDftStages;
            if (pc >= 0 && nc < nch) {
                ok = fch::tc::mbar_wait(&mmab[pc % kDftStages], (uint32_t)((pc / kDftStages) & 1), kTcBound);
                if (ok) {
                    fetch(nc);
                    fetched = nc + 1;
                }
            }
        }
        // the last commit covers every MMA issued; tiles fetched beyond what was consumed (an
        // early stop) are waited for before the CTA's shared memory goes away
        if (issued > 0 && !fch::tc::mbar_wait(&mmab[(issued - 1) % kDftStages],
                                              (uint32_t)(((issued - 1) / kDftStages) & 1), kTcBound))
            ok = false;
        for (int c = issued; c < fetched; c++)
            fch::tc::mbar_wait(&full[c % kDftStages], (uint32_t)((c / kDftStages) & 1), kTcBound);
        ok = ok && issued == nch;
        fch::tc::fence_before_sync();
    }
    ok = __syncthreads_and(ok);
    fch::tc::fence_after_sync();
    if (ok) {
        float v[32];
        fch::tc::tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16), v);
        const long r = row0 + warp * 32 + lane;
        if (r < R) {
            float4 *dst = reinterpret_cast<float4 *>(X + r * 16);
#pragma unroll
            for (int k = 0; k < 8; k++)
                dst[k] = make_float4(v[2 * k], v[16 + 2 * k], v[2 * k + 1], v[16 + 2 * k + 1]);
        }
    } else if (tid == 0) {
        atomicExch(err, 1);
    }
    fch::tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) fch::tc::tmem_dealloc(tmem, 32);
}

// launch of fno_rowdft_tc over R rows of n bf16 at h (n a multiple of 64), with its tensor
// maps and dynamic shared memory (the limit raised once)
cudaError_t launch_rowdft_tc(const __nv_bfloat16 *h, const __nv_bfloat16 *Bt, float2 *X, long R, int n, int *err,
                             cudaStream_t s)
{
    static bool attr = false;
    if (!attr) {
        const cudaError_t e =
            cudaFuncSetAttribute(fno_rowdft_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowdftSmem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    CUtensorMap ma, mb;
    // R rows of n, tiles of 128 rows x 64, zero past the last row; the table's 32 rows x 64
    cudaError_t e = fch_tmap_bf16_2d_sw128(&ma, h, (uint64_t)n, (uint64_t)R, (uint64_t)n * 2, kTcRows);
    if (e == cudaSuccess) e = fch_tmap_bf16_2d_sw128(&mb, Bt, (uint64_t)n, kTcNB, (uint64_t)n * 2, kTcNB);
    if (e != cudaSuccess) return e;
    fno_rowdft_tc<<<(unsigned)((R + kTcRows - 1) / kTcRows), 128, kRowdftSmem, s>>>(ma, mb, X, (int)R, n, err);
    return cudaGetLastError();
}

// Y[f][kyi][kx] = sum_y X[f][y][kx] e^{-2 pi i ky y / n}: one block per (field f, kx).
// The column X[f][.][kx] and the twiddle table (cos, sin)(2 pi j / n) go to shared
// memory; eight threads share each retained ky (thread j of the eight sums the y = j
// mod 8), then three shuffle levels add the eight partial sums in a fixed order.
// n a multiple of 128; dynamic shared memory: 2 n float2.
template <int MM>
__global__ void __launch_bounds__(256) fno_coldft(const float2 *__restrict__ X, const float2 *__restrict__ tw1,
                                                  float2 *__restrict__ Y, int n)
{
    constexpr int K2 = 2 * MM - 1;
    static_assert(K2 <= 32, "eight threads a retained ky in 256 threads");
    extern __shared__ float2 cd_sm[];
    float2 *col = cd_sm, *tw = cd_sm + n;
    const int f = blockIdx.x, kx = blockIdx.y, tid = threadIdx.x;
    for (int y = tid; y < n; y += 256) {
        col[y] = X[((long)f * n + y) * 16 + kx];
        tw[y] = tw1[y];
    }
    __syncthreads();
    const int k = tid >> 3, j = tid & 7; // k = K2 (the last eight threads) computes nothing kept
    const int ky = k < MM ? k : n - (k - MM + 1);
    // the twiddle of y + 8 is the twiddle of y times (cos, sin)(2 pi 8 ky / n): a table
    // read starts each run of 16 such steps (the reads of a warp would meet bank
    // conflicts at stride ky in the table; the products stay within ~16 roundings)
    const float2 step = tw[(8 * ky) & (n - 1)];
    float2 acc = make_float2(0.f, 0.f);
    for (int y0 = j; y0 < n; y0 += 128) {
        float2 w = tw[(ky * y0) & (n - 1)];
#pragma unroll
        for (int r = 0; r < 16; r++) {
            const float2 v = col[y0 + 8 * r];
            acc.x = fmaf(v.x, w.x, fmaf(v.y, w.y, acc.x));
            acc.y = fmaf(v.y, w.x, fmaf(-v.x, w.y, acc.y));
            w = make_float2(fmaf(w.x, step.x, -w.y * step.y), fmaf(w.x, step.y, w.y * step.x));
        }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
    }
    if (j == 0 && k < K2) Y[((long)f * K2 + k) * MM + kx] = acc;
}

// Z[b][o][kyi][kx] = sum_i R[m][o][i] Y[b][i][kyi][kx], m = kx (2M-1) + kyi: one block a
// mode, its weights (contiguous in memory) and channel vectors through shared memory, the
// weight rows padded by one
template <typename WT>
__global__ void __launch_bounds__(128) fno_mix_modes(const float2 *__restrict__ Y, const WT *__restrict__ R,
                                                     float2 *__restrict__ Z, int B, int W, int M)
{
    extern __shared__ __align__(16) float2 mm_smem[];
    float2 *r = mm_smem, *x = mm_smem + W * (W + 1);
    const int K2 = 2 * M - 1, K = M * K2, q = blockIdx.x, kyi = q / M, kx = q - kyi * M;
    const long m = (long)kx * K2 + kyi;
    for (int e = threadIdx.x; e < W * W; e += 128) r[e / W * (W + 1) + e % W] = wld2(R, m * W * W + e);
    for (int b = 0; b < B; b++) {
        __syncthreads(); // the vectors of the sample before are read
        for (int i = threadIdx.x; i < W; i += 128) x[i] = Y[((long)b * W + i) * K + q];
        __syncthreads();
        for (int o = threadIdx.x; o < W; o += 128) {
            float re = 0.f, im = 0.f;
            for (int i = 0; i < W; i++) {
                const float2 v = x[i], w = r[o * (W + 1) + i];
                re += w.x * v.x - w.y * v.y;
                im += w.x * v.y + w.y * v.x;
            }
            Z[((long)b * W + o) * K + q] = make_float2(re, im);
        }
    }
}

// V[f][y][kx] = sum_kyi Z[f][kyi][kx] e^{+2 pi i ky y / n}: one block per (field f, 64
// rows y); Z[f] and the twiddle table (cos, sin)(2 pi j / n) in shared memory, thread
// (y, kx) four outputs. Dynamic shared memory: n float2.
template <int MM>
__global__ void __launch_bounds__(256) fno_icoldft(const float2 *__restrict__ Z, const float2 *__restrict__ tw1,
                                                   float2 *__restrict__ V, long nf, int n)
{
    constexpr int K2 = 2 * MM - 1, YB = 64;
    __shared__ float2 zs[K2 * MM];
    extern __shared__ float2 ic_tw[];
    const int nyb = n / YB;
    const long f = blockIdx.x / nyb;
    const int y0 = (int)(blockIdx.x % nyb) * YB, tid = threadIdx.x;
    for (int i = tid; i < K2 * MM; i += 256) zs[i] = Z[f * K2 * MM + i];
    for (int i = tid; i < n; i += 256) ic_tw[i] = tw1[i];
    __syncthreads();
    for (int i = tid; i < YB * MM; i += 256) {
        const int y = y0 + i / MM, kx = i % MM;
        float re = 0.f, im = 0.f;
#pragma unroll
        for (int k = 0; k < K2; k++) {
            const int ky = k < MM ? k : n - (k - MM + 1);
            const float2 z = zs[k * MM + kx], w = ic_tw[(ky * y) & (n - 1)];
            re = fmaf(z.x, w.x, fmaf(-z.y, w.y, re));
            im = fmaf(z.x, w.y, fmaf(z.y, w.x, im));
        }
        V[(f * n + y) * 16 + kx] = make_float2(re, im);
    }
}

// 8 floats rounded to bfloat16 (nearest even), packed as one 16-byte core row
__device__ __forceinline__ uint4 pack8_bf16(const float *f)
{
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        __nv_bfloat162 b = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
        w[i] = *reinterpret_cast<uint32_t *>(&b);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
// row r, K-core kc of a core-layout tile (see fch_tc.cuh)
__device__ __forceinline__ void core_store(unsigned char *tile, int r, int kc, uint4 v)
{
    *reinterpret_cast<uint4 *>(tile + (r >> 3) * kTcSBO + kc * kTcLBO + (r & 7) * 16) = v;
}

// A operand tiles of 128 points with the points contiguous (core matrices of eight K rows of
// eight points): row k, points 8 xg.. at xg * kMnSBO + (k / 8) * 128 + (k mod 8) * 16, so a
// 16-byte piece of a channel row is stored as it was loaded. kMnSBO: eight K cores and 16
// bytes, which spreads the stores of neighbouring xg over the banks.
constexpr int kMnLBO = 128, kMnSBO = 8 * 128 + 16;
__device__ __forceinline__ void mn_store(unsigned char *tile, int k, int xg, uint4 v)
{
    *reinterpret_cast<uint4 *>(tile + xg * kMnSBO + (k >> 3) * kMnLBO + (k & 7) * 16) = v;
}

// The pointwise layer on the tensor cores: for the 128 points x of a row segment (TMEM lane
// = point), z[o] = sum_j W[o][j] h[j] + b[o] + S[o] with S the inverse x DFT of V, as one
// MMA chain with K = W + 32:
//   A[x][:] = (h[b][j][y][x], j < W | bf16 cos(2 pi kx x/n), kx < 16 | bf16 sin(...))
//   B[o][:] = (W[o][j] | bf16(w(kx)/n^2 Re V[o][y][kx]) | bf16(-w(kx)/n^2 Im V[o][y][kx]))
// D = A B^T (128 x W, FP32 in tensor memory); out = bf16(act(D + b)). h and out are bf16:
// the tensor cores are their only readers, and took them rounded to bf16 from FP32 before,
// so no bit of a result changes while the layer reads and writes half the bytes.
// A CTA takes kPwRows rows y of one segment: the table part of A, the weights in B and the
// tensor memory are set up once, and the next row's activations are loaded while the tensor
// core and the epilogue work on the row before. (One row a CTA with FP32 activations and the
// table read as 32 float2 a thread: 54 us a layer at 1024^2, 32 channels; now 40, the GELU's
// instructions and the row's chain of barriers, MMA and read-back at 20 warps an SM. Rows a
// CTA 2 / 4 / 8 / 16: 471 / 458 / 468 / 484 us a forward pass; no register bound: 475.)
constexpr int kPwRows = 4;
template <int W>
__global__ void __launch_bounds__(128, 5) fno_pw_tc(const __nv_bfloat16 *__restrict__ h, const float2 *__restrict__ V,
                                                 const __nv_bfloat16 *__restrict__ At,
                                                 const __nv_bfloat16 *__restrict__ Wl,
                                                 const __nv_bfloat16 *__restrict__ bl,
                                                 __nv_bfloat16 *__restrict__ out, int n, int act, int *err)
{
    constexpr int K = W + 32, NP = W / 8; // 16-byte pieces of a tile's channels a thread moves
    constexpr int kOutRow = 128 * 2 + 16; // staged output rows, padded
    __shared__ __align__(128) unsigned char sA[16 * kMnSBO];
    __shared__ __align__(128) unsigned char sB[(W / 8) * kTcSBO];
    __shared__ __align__(16) unsigned char sO[W * kOutRow];
    __shared__ float bs[W];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tslot;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int segs = n >> 7, seg = blockIdx.x % segs, y0 = blockIdx.x / segs * kPwRows, b = blockIdx.y;
    const long n2 = (long)n * n;
    if (warp == 0) {
        fch::tc::tmem_alloc(&tslot, 32);
        fch::tc::tmem_relinquish();
    }
    if (tid == 0) {
        fch::tc::mbar_init(&bar, 1);
        fch::tc::mbar_init_fence();
    }
    const int xg = tid & 15, r0 = tid >> 4; // piece i of this thread: channel r0 + 8 i, points 8 xg..
    const long base = (long)b * W * n2 + seg * 128 + 8 * xg;
    // the V part of B: thread (o, kc) rounds eight coefficients of output o, W * 4 threads
    const int vo = tid >> 2, vkc = tid & 3, vpart = vkc >> 1, vk0 = (vkc & 1) * 8;
    const float4 *vp = reinterpret_cast<const float4 *>(V + ((long)b * W + vo) * n * 16 + vk0);
    uint4 hv[NP];
    float4 vv[4];
    auto load = [&](int y) {
#pragma unroll
        for (int i = 0; i < NP; i++)
            hv[i] = *reinterpret_cast<const uint4 *>(h + base + (long)(r0 + 8 * i) * n2 + (long)y * n);
        if (vo < W) {
#pragma unroll
            for (int e = 0; e < 4; e++) vv[e] = vp[(long)y * 8 + e];
        }
    };
    load(y0);
#pragma unroll
    for (int i = 0; i < 4; i++)
        mn_store(sA, W + r0 + 8 * i, xg,
                 *reinterpret_cast<const uint4 *>(At + (long)(r0 + 8 * i) * n + seg * 128 + 8 * xg));
    for (int i = tid; i < W * NP; i += 128) {
        const int o = i / NP, kc = i - o * NP;
        core_store(sB, o, kc, *reinterpret_cast<const uint4 *>(Wl + o * W + kc * 8));
    }
    for (int i = tid; i < W; i += 128) bs[i] = __bfloat162float(bl[i]);
    const float sc = 1.0f / ((float)n * (float)n);
    bool ok = true;
    uint32_t tmem = 0;
    for (int r = 0; r < kPwRows; r++) {
        const int y = y0 + r;
#pragma unroll
        for (int i = 0; i < NP; i++) mn_store(sA, r0 + 8 * i, xg, hv[i]);
        if (vo < W) {
            float f[8];
#pragma unroll
            for (int e = 0; e < 8; e++) {
                const float wk = (vk0 + e == 0 ? 1.f : 2.f) * sc;
                const float4 q = vv[e >> 1];
                f[e] = vpart ? -wk * (e & 1 ? q.w : q.y) : wk * (e & 1 ? q.z : q.x);
            }
            core_store(sB, vo, NP + vkc, pack8_bf16(f));
        }
        fch::tc::fence_async_smem();
        fch::tc::fence_before_sync();
        __syncthreads();
        fch::tc::fence_after_sync();
        tmem = tslot;
        if (tid == 0) {
            constexpr uint32_t idesc = fch::tc::idesc_bf16_f32(128, W, true);
            const uint32_t sa = fch::tc::smem_u32(sA), sb = fch::tc::smem_u32(sB);
#pragma unroll
            for (int k = 0; k < K / 16; k++)
                fch::tc::mma_bf16(tmem, fch::tc::smem_desc(sa + 2 * k * kMnLBO, kMnLBO, kMnSBO),
                                  fch::tc::smem_desc(sb + 2 * k * kTcLBO, kTcLBO, kTcSBO), idesc, k != 0);
            fch::tc::mma_commit(&bar);
        }
        if (r + 1 < kPwRows) load(y + 1);
        ok = __syncthreads_and(fch::tc::mbar_wait(&bar, (uint32_t)(r & 1), kTcBound));
        fch::tc::fence_after_sync();
        if (!ok) break;
        float v[32];
        fch::tc::tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16), v);
#pragma unroll
        for (int o = 0; o < W; o += 2) {
            float2 g2;
            if (act)
                g2 = x2_split(gelu_as2(x2_add(x2(v[o], v[o + 1]), x2(bs[o], bs[o + 1]))));
            else
                g2 = make_float2(v[o] + bs[o], v[o + 1] + bs[o + 1]);
            *reinterpret_cast<__nv_bfloat16 *>(sO + o * kOutRow + tid * 2) = __float2bfloat16_rn(g2.x);
            *reinterpret_cast<__nv_bfloat16 *>(sO + (o + 1) * kOutRow + tid * 2) = __float2bfloat16_rn(g2.y);
        }
        fch::tc::fence_before_sync(); // the accumulator is read before the next row's MMAs
        __syncthreads();
#pragma unroll
        for (int i = 0; i < NP; i++)
            *reinterpret_cast<uint4 *>(out + base + (long)(r0 + 8 * i) * n2 + (long)y * n) =
                *reinterpret_cast<const uint4 *>(sO + (r0 + 8 * i) * kOutRow + xg * 16);
    }
    if (!ok && tid == 0) atomicExch(err, 1);
    fch::tc::fence_before_sync();
    __syncthreads();
    tmem = tslot;
    if (warp == 0) fch::tc::tmem_dealloc(tmem, 32);
}

// The projection on the tensor cores: for 128 points (thread t, TMEM lane t),
// zq = Q1 h + bQ1 as D = A B^T with A[t][:] = h[b][c][p] in bf16 (K = W) and
// B = Q1 (W2 x W), then y = bQ2 + sum_d Q2[d] GELU(zq[d]) in the epilogue. A tile's points
// lie in one sample (n a multiple of 128).
template <int W>
__global__ void __launch_bounds__(128) fno_proj_tc(const __nv_bfloat16 *__restrict__ h,
                                                   const __nv_bfloat16 *__restrict__ Q1,
                                                   const __nv_bfloat16 *__restrict__ bQ1,
                                                   const __nv_bfloat16 *__restrict__ Q2,
                                                   const __nv_bfloat16 *__restrict__ bQ2, float *__restrict__ y,
                                                   int n2, int W2, int *err)
{
    __shared__ __align__(128) unsigned char sA[16 * kMnSBO];
    __shared__ __align__(128) unsigned char sB[(kMaxW2 / 8) * kTcSBO];
    __shared__ __align__(16) float bq[kMaxW2], q2[kMaxW2];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tslot;
    const int tid = threadIdx.x, warp = tid >> 5;
    const long g0 = (long)blockIdx.x * 128, b = g0 / n2, p0 = g0 - b * n2;
    const uint32_t ncols = W2 <= 32 ? 32 : (W2 <= 64 ? 64 : 128);
    if (warp == 0) {
        fch::tc::tmem_alloc(&tslot, ncols);
        fch::tc::tmem_relinquish();
    }
    if (tid == 0) {
        fch::tc::mbar_init(&bar, 1);
        fch::tc::mbar_init_fence();
    }
    const int xg = tid & 15, r0 = tid >> 4;
#pragma unroll
    for (int i = 0; i < W / 8; i++)
        mn_store(sA, r0 + 8 * i, xg,
                 __ldcs(reinterpret_cast<const uint4 *>(h + (b * W + r0 + 8 * i) * n2 + p0 + 8 * xg)));
    for (int i = tid; i < W2 * (W / 8); i += 128) {
        const int d = i / (W / 8), kc = i - d * (W / 8);
        core_store(sB, d, kc, *reinterpret_cast<const uint4 *>(Q1 + d * W + kc * 8));
    }
    for (int i = tid; i < W2; i += 128) {
        bq[i] = __bfloat162float(bQ1[i]);
        q2[i] = __bfloat162float(Q2[i]);
    }
    fch::tc::fence_async_smem();
    fch::tc::fence_before_sync();
    __syncthreads();
    fch::tc::fence_after_sync();
    const uint32_t tmem = tslot;
    if (tid == 0) {
        const uint32_t idesc = fch::tc::idesc_bf16_f32(128, W2, true);
        const uint32_t sa = fch::tc::smem_u32(sA), sb = fch::tc::smem_u32(sB);
#pragma unroll
        for (int k = 0; k < W / 16; k++)
            fch::tc::mma_bf16(tmem, fch::tc::smem_desc(sa + 2 * k * kMnLBO, kMnLBO, kMnSBO),
                              fch::tc::smem_desc(sb + 2 * k * kTcLBO, kTcLBO, kTcSBO), idesc, k != 0);
        fch::tc::mma_commit(&bar);
    }
    const bool ok = __syncthreads_and(fch::tc::mbar_wait(&bar, 0, kTcBound));
    fch::tc::fence_after_sync();
    if (ok) {
        // W2 is a multiple of 16: sixteen accumulator columns at a time, the biases and
        // the second layer's weights four at a time from shared memory
        f32x2 acc = x2(__bfloat162float(bQ2[0]), 0.f); // two partial sums, added at the end
        for (int c0 = 0; c0 < W2; c0 += 16) {
            float v[16];
            fch::tc::tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
            for (int d = 0; d < 16; d += 4) {
                const float4 b4 = *reinterpret_cast<const float4 *>(bq + c0 + d);
                const float4 q4 = *reinterpret_cast<const float4 *>(q2 + c0 + d);
                acc = x2_fma(x2(q4.x, q4.y), gelu_as2(x2_add(x2(v[d], v[d + 1]), x2(b4.x, b4.y))), acc);
                acc = x2_fma(x2(q4.z, q4.w), gelu_as2(x2_add(x2(v[d + 2], v[d + 3]), x2(b4.z, b4.w))), acc);
            }
        }
        const float2 a2 = x2_split(acc);
        y[g0 + tid] = a2.x + a2.y;
    } else if (tid == 0) {
        atomicExch(err, 1);
    }
    fch::tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) fch::tc::tmem_dealloc(tmem, ncols);
}

// dY[b][o][m] (compact, K modes a field) = H(w(kx)/n^2 Fd(m)), Fd = R2C of the
// spectral branch's output gradient
__global__ void fno_dY(const float2 *__restrict__ Fd, float2 *__restrict__ dY, int B, int W, int M, int n)
{
    const int K2 = 2 * M - 1, K = M * K2;
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)B * W * K) return;
    const int m = (int)(t % K);
    const long f = t / K;
    const long S = (long)(n / 2 + 1) * n;
    const int kx = m / K2, kyi = m % K2, ky = mode_ky(kyi, M, n);
    const float inv = 1.0f / ((float)n * (float)n);
    const float2 *F = Fd + f * S;
    float2 v;
    if (kx == 0) {
        const float2 a = F[ky], c = F[(n - ky) % n]; // w = 1 at kx = 0
        v = make_float2(0.5f * (a.x + c.x) * inv, 0.5f * (a.y - c.y) * inv);
    } else {
        const float2 a = F[(long)kx * n + ky];
        v = make_float2(2.f * a.x * inv, 2.f * a.y * inv);
    }
    dY[t] = v;
}

// dR[m][o][i] = sum_b dY[b][o][m] conj(X[b][i](m))
__global__ void fno_dR(const float2 *__restrict__ dY, const float2 *__restrict__ X, float2 *__restrict__ dR,
                       int B, int W, int M, int n)
{
    const int K2 = 2 * M - 1, K = M * K2;
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)K * W * W) return;
    const int i = (int)(t % W), o = (int)((t / W) % W), m = (int)(t / ((long)W * W));
    const long S = (long)(n / 2 + 1) * n;
    const int kx = m / K2, ky = mode_ky(m % K2, M, n);
    float re = 0.f, im = 0.f;
    for (int b = 0; b < B; b++) {
        const float2 d = dY[((long)b * W + o) * K + m];
        const float2 x = X[((long)b * W + i) * S + (long)kx * n + ky];
        re += d.x * x.x + d.y * x.y;
        im += d.y * x.x - d.x * x.y;
    }
    dR[t] = make_float2(re, im);
}

// Z[b W + i](m) = n^2 v(kx) sum_o conj(R[m][o][i]) dY[b][o][m], through H at kx = 0,
// so that C2R(Z) is the gradient of the layer input through the spectral branch
__global__ void fno_dX(const float2 *__restrict__ dY, const float2 *__restrict__ R, float2 *__restrict__ Z,
                       int B, int W, int M, int n)
{
    const int K2 = 2 * M - 1, K = M * K2;
    const int items = M + (M - 1) * K2;
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)B * W * items) return;
    const int it = (int)(t % items), i = (int)((t / items) % W), b = (int)(t / ((long)items * W));
    const long S = (long)(n / 2 + 1) * n;
    const float n2 = (float)n * (float)n;
    auto back = [&](int m) {
        float re = 0.f, im = 0.f;
        for (int o = 0; o < W; o++) {
            const float2 d = dY[((long)b * W + o) * K + m];
            const float2 w = R[((long)m * W + o) * W + i];
            re += w.x * d.x + w.y * d.y;
            im += w.x * d.y - w.y * d.x;
        }
        return make_float2(re, im);
    };
    float2 *Zf = Z + ((long)b * W + i) * S;
    if (it < M) { // kx = 0, v = 1
        const int ky = it;
        const float2 dp = back(ky);
        if (ky == 0) {
            Zf[0] = make_float2(n2 * dp.x, 0.f);
        } else {
            const float2 dm = back(ky + M - 1);
            const float2 hh = make_float2(0.5f * n2 * (dp.x + dm.x), 0.5f * n2 * (dp.y - dm.y));
            Zf[ky] = hh;
            Zf[n - ky] = make_float2(hh.x, -hh.y);
        }
    } else { // v = 1/2
        const int j = it - M, kx = 1 + j / K2, kyi = j % K2;
        const float2 d = back(kx * K2 + kyi);
        Zf[(long)kx * n + mode_ky(kyi, M, n)] = make_float2(0.5f * n2 * d.x, 0.5f * n2 * d.y);
    }
}

// The products over the channels at one retained mode (block m) on mode-major spectra
// [m][b W + c]: Y[b][o] = sum_i R[o][i] X[b][i]. The weights pass through shared memory, rows
// padded by one (lanes read consecutive o).
template <typename WT>
__global__ void __launch_bounds__(256) fno_mode_mix(const float2 *__restrict__ X, const WT *__restrict__ R,
                                                    float2 *__restrict__ Y, int BW, int W)
{
    extern __shared__ __align__(16) float2 mm_smem[];
    float2 *r = mm_smem, *x = mm_smem + W * (W + 1);
    const long m = blockIdx.x;
    for (int e = threadIdx.x; e < W * W; e += 256) r[e / W * (W + 1) + e % W] = wld2(R, m * W * W + e);
    for (int e = threadIdx.x; e < BW; e += 256) x[e] = X[m * BW + e];
    __syncthreads();
    for (int e = threadIdx.x; e < BW; e += 256) {
        const float2 *ro = r + e % W * (W + 1), *xb = x + e / W * W;
        float re = 0.f, im = 0.f;
        for (int i = 0; i < W; i++) {
            const float2 w = ro[i], v = xb[i];
            re += w.x * v.x - w.y * v.y;
            im += w.x * v.y + w.y * v.x;
        }
        Y[m * BW + e] = make_float2(re, im);
    }
}

// Backward at one mode: dR[o][i] = sum_b dY[b][o] conj X[b][i] and
// Z[b][i] = sum_o conj(R[o][i]) dY[b][o].
__global__ void __launch_bounds__(256) fno_mode_bwd(const float2 *__restrict__ dY, const float2 *__restrict__ X,
                                                    const float2 *__restrict__ R, float2 *__restrict__ dR,
                                                    float2 *__restrict__ Z, int BW, int W)
{
    extern __shared__ __align__(16) float2 mm_smem[];
    float2 *r = mm_smem, *x = r + W * W, *d = x + BW;
    const long m = blockIdx.x;
    for (int e = threadIdx.x; e < W * W; e += 256) r[e] = R[m * W * W + e];
    for (int e = threadIdx.x; e < BW; e += 256) {
        x[e] = X[m * BW + e];
        d[e] = dY[m * BW + e];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < W * W; e += 256) {
        const int o = e / W, i = e % W;
        float re = 0.f, im = 0.f;
        for (int b = 0; b < BW; b += W) {
            const float2 u = d[b + o], v = x[b + i];
            re += u.x * v.x + u.y * v.y;
            im += u.y * v.x - u.x * v.y;
        }
        dR[m * W * W + e] = make_float2(re, im);
    }
    for (int e = threadIdx.x; e < BW; e += 256) {
        const int i = e % W, b = e - i;
        float re = 0.f, im = 0.f;
        for (int o = 0; o < W; o++) {
            const float2 w = r[o * W + i], u = d[b + o];
            re += w.x * u.x + w.y * u.y;
            im += w.x * u.y - w.y * u.x;
        }
        Z[m * BW + e] = make_float2(re, im);
    }
}

__global__ void fno_add(float *__restrict__ a, const float *__restrict__ b, long cnt)
{
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < cnt) a[t] += b[t];
}

// Weight-gradient partials of a dense layer: G[a][c] = sum over points of A(a, pt) Bm(c, pt)
// and the bias row sums of A, with A(a, (b, p)) = A[(b na + a) n2 + p] (Bm alike). A block
// takes the 32 x 32 outputs (32 blockIdx.y, 32 blockIdx.z) over its share of the points,
// staged 64 at a time in shared memory (rows padded to 68 floats: the 16-byte reads of eight
// lanes fall on distinct banks); a thread owns 4 x 4 outputs of one quarter of the points,
// 64 fused multiply-adds per eight 16-byte reads, and the quarters are summed at the end.
// Block k writes part[k][off + a nb + c] and part[k][off + na nb + a].
// The kernel before gave a thread 1-8 outputs with one multiply-add per two scalar reads, and
// the sums of 1024 partials ran in one to eight blocks: at 128^2, batch 8, 32 channels, 1.17 ms
// of partials and 0.85 ms of sums a training step.
constexpr int kWgPts = 64, kWgPad = kWgPts + 4;
__global__ void __launch_bounds__(256) fno_wgrad_part(const float *__restrict__ A, int na,
                                                      const float *__restrict__ Bm, int nb, int n2, long npts,
                                                      int chunk, float *__restrict__ part, long stride, long off)
{
    __shared__ __align__(16) float sm[2 * 32 * kWgPad]; // then the quarters' sums [4][32 * 33]
    static_assert(2 * 32 * kWgPad >= 4 * 32 * 33, "the sums fit the stage");
    float(*acc_sm)[32 * 33] = (float(*)[32 * 33])sm;
    float *sa = sm, *sb = sm + 32 * kWgPad;
    const int tid = threadIdx.x, kg = tid >> 6, ta = (tid >> 3) & 7, tc = tid & 7;
    const int a0 = blockIdx.y * 32, c0 = blockIdx.z * 32;
    const int lr = tid >> 3, lk = (tid & 7) * 4; // the row and points this thread stages
    const bool la = a0 + lr < na, lb = c0 + lr < nb;
    float acc[4][4], bias[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        bias[i] = 0.f;
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = 0.f;
    }
    const long p0 = (long)blockIdx.x * chunk, p1 = min(p0 + chunk, npts);
    // a stage's points lie within one sample (n2 is a multiple of 256)
    const bool vec = !((uintptr_t)Bm & 15); // the network's input is the caller's array
    auto fetch = [&](long q, float4 *fa, float4 *fb) {
        const long b = q / n2, p = q - b * n2 + lk;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        const float *pa = A + (b * na + a0 + lr) * n2 + p, *pb = Bm + (b * nb + c0 + lr) * n2 + p;
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const float *w = pb + 32 * h;
            fa[h] = la ? *(const float4 *)(pa + 32 * h) : zero;
            fb[h] = !lb ? zero : vec ? *(const float4 *)w : make_float4(w[0], w[1], w[2], w[3]);
        }
    };
    float4 fa[2], fb[2];
    if (p0 < p1) fetch(p0, fa, fb);
    for (long q = p0; q < p1; q += kWgPts) {
        __syncthreads();
#pragma unroll
        for (int h = 0; h < 2; h++) {
            *(float4 *)(sa + lr * kWgPad + lk + 32 * h) = fa[h];
            *(float4 *)(sb + lr * kWgPad + lk + 32 * h) = fb[h];
        }
        __syncthreads();
        if (q + kWgPts < p1) fetch(q + kWgPts, fa, fb);
#pragma unroll
        for (int h = 0; h < kWgPts / 16; h++) {
            const int k = kg * (kWgPts / 4) + h * 4;
            float4 va[4], vb[4];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                va[i] = *(const float4 *)(sa + (ta + 8 * i) * kWgPad + k);
                vb[i] = *(const float4 *)(sb + (tc + 8 * i) * kWgPad + k);
            }
#pragma unroll
            for (int i = 0; i < 4; i++) {
                bias[i] += (va[i].x + va[i].y) + (va[i].z + va[i].w);
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    float v = acc[i][j];
                    v = fmaf(va[i].x, vb[j].x, v);
                    v = fmaf(va[i].y, vb[j].y, v);
                    v = fmaf(va[i].z, vb[j].z, v);
                    acc[i][j] = fmaf(va[i].w, vb[j].w, v);
                }
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; i++) {
#pragma unroll
        for (int j = 0; j < 4; j++) acc_sm[kg][(ta + 8 * i) * 33 + tc + 8 * j] = acc[i][j];
        if (tc == 0) acc_sm[kg][(ta + 8 * i) * 33 + 32] = bias[i];
    }
    __syncthreads();
    float *out = part + blockIdx.x * stride + off;
    for (int e = tid; e < 32 * 33; e += 256) {
        const int a = a0 + e / 33, j = e % 33, c = c0 + j;
        const float v = (acc_sm[0][e] + acc_sm[1][e]) + (acc_sm[2][e] + acc_sm[3][e]);
        if (a >= na) continue;
        if (j == 32) {
            if (blockIdx.z == 0) out[(long)na * nb + a] = v;
        } else if (c < nb) {
            out[(long)a * nb + c] = v;
        }
    }
}

// The sums of all layers' partials, one launch: column o of part[nblk][stride] into its
// parameter's gradient (runs of consecutive parameters: part offset, length, destination).
constexpr int kWgRuns = 18; // lift, up to sixteen layers, projection
struct WgRuns {
    int n;
    long off[kWgRuns];
    long len[kWgRuns];
    float *dst[kWgRuns];
};
__global__ void __launch_bounds__(256) fno_wgrad_sum(const float *__restrict__ part, int nblk, long stride,
                                                     const WgRuns runs)
{
    __shared__ float sm[8][32];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const long o = (long)blockIdx.x * 32 + lane;
    float v = 0.f;
    if (o < stride) {
#pragma unroll 4
        for (int k = g; k < nblk; k += 8) v += part[k * stride + o];
    }
    sm[g][lane] = v;
    __syncthreads();
    if (g == 0 && o < stride) {
        v = ((sm[0][lane] + sm[1][lane]) + (sm[2][lane] + sm[3][lane])) +
            ((sm[4][lane] + sm[5][lane]) + (sm[6][lane] + sm[7][lane]));
        for (int r = 0; r < runs.n; r++)
            if (o >= runs.off[r] && o < runs.off[r] + runs.len[r]) runs.dst[r][o - runs.off[r]] = v;
    }
}

// sums of squared residuals in double, one partial a block (the host adds them)
constexpr int kLossBlocks = 256;
__global__ void __launch_bounds__(256) fno_loss_part(const float *__restrict__ sq, long cnt, double *__restrict__ part)
{
    __shared__ double sm[8];
    double v = 0;
    for (long i = (long)blockIdx.x * 256 + threadIdx.x; i < cnt; i += (long)gridDim.x * 256) v += (double)sq[i];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0;
        for (int w = 0; w < 8; w++) t += sm[w];
        part[blockIdx.x] = t;
    }
}

// Adam (Kingma & Ba), bias-corrected, on the flat parameter vector
__global__ void fno_adam(float *__restrict__ w, const float *__restrict__ g, float *__restrict__ m,
                         float *__restrict__ v, long cnt, float lr, float b1, float b2, float eps, float c1, float c2)
{
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= cnt) return;
    const float gg = g[t];
    const float mm = b1 * m[t] + (1.f - b1) * gg;
    const float vv = b2 * v[t] + (1.f - b2) * gg * gg;
    m[t] = mm;
    v[t] = vv;
    w[t] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
}

} // namespace

struct fch_fno {
    int W, L, M, W2, cin, K;
    cudaStream_t stream;
    size_t np;
    float *params, *grads, *am, *av;
    long long adam_t;
    // per (B, n) buffers
    int B, n;
    fch_fft_plan *plan;
    float *h;     // (L + 1) x [B][W][n^2]
    float *z;     // L x [B][W][n^2]
    // spectra: up to 256^2 the retained modes only, mode-major (fch_fnomodes.cuh): X L x
    // [K][B W], Ysp and dY [K][B W]; on larger grids (or M > 32) X L x [B W][(n/2+1) n], Ysp
    // and Fd [B W][(n/2+1) n] (Ysp zero outside the retained modes), dY [B][W][K]
    bool modes;
    float2 *X, *Ysp, *Fd, *dY;
    float *s;     // [B][W][n^2]
    float *dh, *dz, *tmp; // [B][W][n^2]
    float *q, *dzq;       // [B][W2][n^2]
    float *y, *dy, *sq;   // [B][n^2]
    float *part;          // weight-gradient partials
    double *lpart;        // the loss's partial sums
    const float *a;       // the last forward pass's input
    bool have_fwd;
    __nv_bfloat16 *pbf;   // bfloat16 copy of params (fch_fno_set_bf16), else null
    bool fwd_bf16;        // the last forward pass read the bfloat16 copy
    // truncated-DFT spectral convolutions (fch_fno_set_bf16(f, 2)): tables for tc_n,
    // work arrays for (tc_B, tc_n), the device error flag of the tensor-core kernel
    bool tc;
    int tc_B, tc_n;
    __nv_bfloat16 *tc_Bt, *tc_At; // [32][n]
    __nv_bfloat16 *tc_h[2];       // [B][W][n^2]: a layer's input and output
    float2 *tc_tw;        // [16][n]
    float2 *tc_X, *tc_V;  // [B W n][16]
    float2 *tc_Y, *tc_Z;  // [B W][2M-1][M]
    int *tc_err;
    double *hsum;
    char err[256];
};

namespace {

size_t offset_of(const fch_fno *f, int what, int l)
{
    // what: 0 P, 1 bP, 2 W_l, 3 b_l, 4 R_l, 5 Q1, 6 bQ1, 7 Q2, 8 bQ2
    const size_t W = f->W, lay = W * W + W + (size_t)f->K * W * W * 2;
    const size_t base = W * f->cin + W;
    switch (what) {
    case 0: return 0;
    case 1: return W * f->cin;
    case 2: return base + l * lay;
    case 3: return base + l * lay + W * W;
    case 4: return base + l * lay + W * W + W;
    case 5: return base + f->L * lay;
    case 6: return base + f->L * lay + (size_t)f->W2 * W;
    case 7: return base + f->L * lay + (size_t)f->W2 * W + f->W2;
    default: return base + f->L * lay + (size_t)f->W2 * W + 2 * f->W2;
    }
}

// blocks the points of a weight gradient are split over (two an SM of the 152 at the most,
// whole stages), and the partial sums of all layers in one block's row
int wgrad_blocks(long npts, int &chunk)
{
    const long runs = npts / kWgPts, per = (runs + 303) / 304;
    chunk = (int)(per * kWgPts);
    return (int)((runs + per - 1) / per);
}
size_t wgrad_stride(const fch_fno *f)
{
    return (size_t)f->W * f->cin + f->W + (size_t)f->L * (f->W * f->W + f->W) + (size_t)f->W2 * f->W + 2 * f->W2 + 1;
}

// whether the spectral branch runs on the retained modes inside a block: grids whose rows and
// kept columns fit an SM's shared memory twice, and channel vectors of a mode that fit the
// products' 48 KB
bool modes_fit(const fch_fno *f, int B, int n)
{
    return n >= 32 && n <= 256 && f->M <= 32 && (size_t)B * f->W <= 2048;
}

template <int LOGN>
cudaError_t field_modes_t(fch_fno *f, const float *h, float2 *out, float s0, float s1, int herm)
{
    typedef fch::FnoModes<LOGN> G;
    cudaError_t e = cudaFuncSetAttribute(fch::fno_field_modes<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         G::smem(32));
    if (e != cudaSuccess) return e;
    fch::fno_field_modes<LOGN><<<f->B * f->W, G::threads, G::smem(f->M), f->stream>>>(
        h, out, (const float2 *)fch_fft_plan_twiddles(f->plan), f->M, s0, s1, herm);
    return cudaGetLastError();
}
cudaError_t field_modes(fch_fno *f, const float *h, float2 *out, float s0, float s1, int herm)
{
    switch (f->n) {
    case 32: return field_modes_t<5>(f, h, out, s0, s1, herm);
    case 64: return field_modes_t<6>(f, h, out, s0, s1, herm);
    case 128: return field_modes_t<7>(f, h, out, s0, s1, herm);
    case 256: return field_modes_t<8>(f, h, out, s0, s1, herm);
    }
    return cudaErrorInvalidValue;
}
template <int LOGN>
cudaError_t modes_field_t(fch_fno *f, const float2 *Y, const float *base, float *out, float s0, float s1)
{
    typedef fch::FnoModes<LOGN> G;
    cudaError_t e = cudaFuncSetAttribute(fch::fno_modes_field<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         G::smem(32));
    if (e != cudaSuccess) return e;
    fch::fno_modes_field<LOGN><<<f->B * f->W, G::threads, G::smem(f->M), f->stream>>>(
        Y, base, out, (const float2 *)fch_fft_plan_twiddles(f->plan), f->M, s0, s1);
    return cudaGetLastError();
}
cudaError_t modes_field(fch_fno *f, const float2 *Y, const float *base, float *out, float s0, float s1)
{
    switch (f->n) {
    case 32: return modes_field_t<5>(f, Y, base, out, s0, s1);
    case 64: return modes_field_t<6>(f, Y, base, out, s0, s1);
    case 128: return modes_field_t<7>(f, Y, base, out, s0, s1);
    case 256: return modes_field_t<8>(f, Y, base, out, s0, s1);
    }
    return cudaErrorInvalidValue;
}

void free_buffers(fch_fno *f)
{
    void *bufs[] = {f->h, f->z, f->X, f->Ysp, f->Fd, f->dY, f->s, f->dh, f->dz, f->tmp,
                    f->q, f->dzq, f->y, f->dy, f->sq, f->part, f->lpart};
    for (void *b : bufs)
        if (b) cudaFree(b);
    f->h = f->z = f->s = f->dh = f->dz = f->tmp = f->q = f->dzq = f->y = f->dy = f->sq = f->part = nullptr;
    f->lpart = nullptr;
    f->X = f->Ysp = f->Fd = f->dY = nullptr;
    if (f->plan) fch_fft_plan_destroy(f->plan);
    f->plan = nullptr;
    f->B = f->n = 0;
    f->have_fwd = false;
}

fch_status ensure_buffers(fch_fno *f, int B, int n)
{
    if (f->B == B && f->n == n) return FCH_OK;
    free_buffers(f);
    const size_t n2 = (size_t)n * n, fld = (size_t)B * f->W * n2, S = (size_t)(n / 2 + 1) * n;
    cudaError_t e = cudaSuccess;
    auto al = [&](void **p, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(p, bytes);
    };
    al((void **)&f->h, (f->L + 1) * fld * 4);
    al((void **)&f->z, f->L * fld * 4);
    f->modes = modes_fit(f, B, n);
    const size_t spec = (size_t)B * f->W * (f->modes ? (size_t)f->K : S) * 8;
    al((void **)&f->X, f->L * spec);
    al((void **)&f->Ysp, spec);
    if (!f->modes) al((void **)&f->Fd, spec);
    al((void **)&f->dY, (size_t)B * f->W * f->K * 8);
    al((void **)&f->s, fld * 4);
    al((void **)&f->dh, fld * 4);
    al((void **)&f->dz, fld * 4);
    al((void **)&f->tmp, fld * 4);
    al((void **)&f->q, (size_t)B * f->W2 * n2 * 4);
    al((void **)&f->dzq, (size_t)B * f->W2 * n2 * 4);
    al((void **)&f->y, (size_t)B * n2 * 4);
    al((void **)&f->dy, (size_t)B * n2 * 4);
    al((void **)&f->sq, (size_t)B * n2 * 4);
    int chunk;
    al((void **)&f->part, (size_t)wgrad_blocks((long)B * n2, chunk) * wgrad_stride(f) * 4);
    al((void **)&f->lpart, kLossBlocks * sizeof(double));
    if (e == cudaSuccess && !f->modes) e = cudaMemsetAsync(f->Ysp, 0, spec, f->stream);
    if (e != cudaSuccess) {
        snprintf(f->err, sizeof(f->err), "fch_fno: %s", cudaGetErrorString(e));
        cudaGetLastError(); // reported here: the next launch's check does not meet it again
        free_buffers(f);
        return e == cudaErrorMemoryAllocation ? FCH_ENOMEM : FCH_ECUDA;
    }
    fch_status s = fch_fft_plan_create(n, 1, f->stream, &f->plan);
    if (s != FCH_OK) {
        free_buffers(f);
        return s;
    }
    f->B = B;
    f->n = n;
    return FCH_OK;
}

inline unsigned grid(long cnt, int bs) { return (unsigned)((cnt + bs - 1) / bs); }

// launch kernel<W> for the channel count W (8, 16 or 32)
#define WDISPATCH(Wv, kern, g, b, st, ...)                                                          \
    do {                                                                                           \
        if ((Wv) == 8)                                                                             \
            kern<8><<<(g), (b), 0, (st)>>>(__VA_ARGS__);                                           \
        else if ((Wv) == 16)                                                                       \
            kern<16><<<(g), (b), 0, (st)>>>(__VA_ARGS__);                                          \
        else                                                                                       \
            kern<32><<<(g), (b), 0, (st)>>>(__VA_ARGS__);                                          \
    } while (0)

// the same for a kernel templated on the channel count and the weight type
#define WDISPATCH_T(Wv, kern, WT, g, b, st, ...)                                                   \
    do {                                                                                           \
        if ((Wv) == 8)                                                                             \
            kern<8, WT><<<(g), (b), 0, (st)>>>(__VA_ARGS__);                                       \
        else if ((Wv) == 16)                                                                       \
            kern<16, WT><<<(g), (b), 0, (st)>>>(__VA_ARGS__);                                      \
        else                                                                                       \
            kern<32, WT><<<(g), (b), 0, (st)>>>(__VA_ARGS__);                                      \
    } while (0)

// partials of G[na][nb] = sum_points A Bm^T and of the row sums of A at offset off
cudaError_t wgrad(fch_fno *f, const float *A, int na, const float *Bm, int nb, long off)
{
    const long npts = (long)f->B * f->n * f->n;
    int chunk;
    const int nblk = wgrad_blocks(npts, chunk);
    fno_wgrad_part<<<dim3(nblk, (na + 31) / 32, (nb + 31) / 32), 256, 0, f->stream>>>(
        A, na, Bm, nb, f->n * f->n, npts, chunk, f->part, (long)wgrad_stride(f), off);
    return cudaGetLastError();
}

} // namespace

cudaStream_t fch_fno_stream_of(const fch_fno *f) { return f->stream; }

extern "C" fch_status fch_fno_create(int width, int layers, int modes, int proj, void *stream, fch_fno **out)
{
    if (!out || (width != 8 && width != 16 && width != 32) || layers < 1 || layers > 16 || modes < 1 ||
        proj < 1 || proj > kMaxW2 || proj * width > kMaxQ1) {
        fch_set_thread_error("fch_fno_create: invalid argument");
        return FCH_EINVAL;
    }
    fch_fno *f = (fch_fno *)calloc(1, sizeof(fch_fno));
    if (!f) return FCH_ENOMEM;
    f->W = width;
    f->L = layers;
    f->M = modes;
    f->W2 = proj;
    f->cin = 2;
    f->K = modes * (2 * modes - 1);
    f->stream = (cudaStream_t)stream;
    f->np = offset_of(f, 8, 0) + 1;
    cudaError_t e = cudaMalloc((void **)&f->params, f->np * 4);
    if (e == cudaSuccess) e = cudaMalloc((void **)&f->grads, f->np * 4);
    if (e == cudaSuccess) e = cudaMalloc((void **)&f->am, f->np * 4);
    if (e == cudaSuccess) e = cudaMalloc((void **)&f->av, f->np * 4);
    if (e == cudaSuccess) e = cudaMallocHost((void **)&f->hsum, kLossBlocks * sizeof(double));
    if (e == cudaSuccess) e = cudaMemsetAsync(f->params, 0, f->np * 4, f->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(f->grads, 0, f->np * 4, f->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(f->am, 0, f->np * 4, f->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(f->av, 0, f->np * 4, f->stream);
    if (e != cudaSuccess) {
        fch_set_thread_error(cudaGetErrorString(e));
        cudaGetLastError();
        fch_fno_destroy(f);
        return FCH_ECUDA;
    }
    *out = f;
    return FCH_OK;
}

extern "C" fch_status fch_fno_destroy(fch_fno *f)
{
    if (!f) return FCH_OK;
    if (f->stream) cudaStreamSynchronize(f->stream);
    free_buffers(f);
    for (void *b : {(void *)f->params, (void *)f->grads, (void *)f->am, (void *)f->av, (void *)f->pbf,
                    (void *)f->tc_Bt, (void *)f->tc_At, (void *)f->tc_h[0], (void *)f->tc_h[1], (void *)f->tc_tw, (void *)f->tc_X, (void *)f->tc_V, (void *)f->tc_Y,
                    (void *)f->tc_Z, (void *)f->tc_err})
        if (b) cudaFree(b);
    if (f->hsum) cudaFreeHost(f->hsum);
    free(f);
    return FCH_OK;
}

extern "C" fch_status fch_fno_num_params(const fch_fno *f, size_t *count)
{
    if (!f || !count) return FCH_EINVAL;
    *count = f->np;
    return FCH_OK;
}

static fch_status refresh_bf16(fch_fno *f);

static fch_status copy_vec(fch_fno *f, float *dev, const float *src_host, float *dst_host, size_t cnt)
{
    if (!f || cnt != f->np) return FCH_EINVAL;
    cudaError_t e = src_host ? cudaMemcpyAsync(dev, src_host, cnt * 4, cudaMemcpyHostToDevice, f->stream)
                             : cudaMemcpyAsync(dst_host, dev, cnt * 4, cudaMemcpyDeviceToHost, f->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(f->stream);
    return e == cudaSuccess ? FCH_OK : FCH_ECUDA;
}

extern "C" fch_status fch_fno_set_params(fch_fno *f, const float *host, size_t cnt)
{
    if (!host) return FCH_EINVAL;
    fch_status s = copy_vec(f, f ? f->params : nullptr, host, nullptr, cnt);
    if (s == FCH_OK) {
        cudaMemsetAsync(f->am, 0, f->np * 4, f->stream);
        cudaMemsetAsync(f->av, 0, f->np * 4, f->stream);
        f->adam_t = 0;
        s = refresh_bf16(f);
    }
    return s;
}

extern "C" fch_status fch_fno_get_params(fch_fno *f, float *host, size_t cnt)
{
    if (!host) return FCH_EINVAL;
    return copy_vec(f, f ? f->params : nullptr, nullptr, host, cnt);
}

extern "C" fch_status fch_fno_get_grads(fch_fno *f, float *host, size_t cnt)
{
    if (!host) return FCH_EINVAL;
    return copy_vec(f, f ? f->grads : nullptr, nullptr, host, cnt);
}

static fch_status spec_error(fch_fno *f, cudaError_t e)
{
    snprintf(f->err, sizeof(f->err), "fch_fno (spectral branch): %s", cudaGetErrorString(e));
    fch_set_thread_error(f->err);
    return FCH_ECUDA;
}

// the forward pass with weights P of type WT (FP32 parameters or their bfloat16 copy)
template <typename WT>
static fch_status forward_impl(fch_fno *f, int batch, int n, const float *a, float *y, const WT *P)
{
    fch_status st = ensure_buffers(f, batch, n);
    if (st != FCH_OK) return st;
    const int W = f->W, n2 = n * n;
    const long pts = (long)batch * n2;
    const size_t fld = (size_t)batch * W * n2, S = (size_t)(n / 2 + 1) * n;
    cudaStream_t s = f->stream;
    {
        const WT *P0 = P + offset_of(f, 0, 0), *P1 = P + offset_of(f, 1, 0);
        if (W == 8)
            fno_lift_t<WT, 8, 2><<<grid(pts, 256), 256, 0, s>>>(a, P0, P1, f->h, pts, n2);
        else if (W == 16)
            fno_lift_t<WT, 16, 2><<<grid(pts, 256), 256, 0, s>>>(a, P0, P1, f->h, pts, n2);
        else
            fno_lift_t<WT, 32, 2><<<grid(pts, 256), 256, 0, s>>>(a, P0, P1, f->h, pts, n2);
    }
    for (int l = 0; l < f->L; l++) {
        float *hin = f->h + l * fld, *hout = f->h + (l + 1) * fld;
        const WT *R = P + offset_of(f, 4, l);
        if (f->modes) {
            float2 *X = f->X + (size_t)l * batch * W * f->K;
            const int BW = batch * W, smem = (W * (W + 1) + BW) * 8;
            cudaError_t e = field_modes(f, hin, X, 1.f, 1.f, 0);
            if (e == cudaSuccess) {
                fno_mode_mix<WT><<<f->K, 256, smem, s>>>(X, R, f->Ysp, BW, W);
                const float inv = 1.0f / ((float)n * (float)n);
                e = modes_field(f, f->Ysp, nullptr, f->s, inv, inv);
            }
            if (e != cudaSuccess) return spec_error(f, e);
        } else {
            float2 *X = f->X + (size_t)l * batch * W * S;
            if ((st = fch_fft_r2c(f->plan, hin, X, batch * W)) != FCH_OK) return st;
            const int items = f->M + (f->M - 1) * (2 * f->M - 1);
            fno_mix<WT><<<grid((long)batch * W * items, 256), 256, 0, s>>>(X, R, f->Ysp, batch, W, f->M, n);
            if ((st = fch_fft_c2r(f->plan, f->Ysp, f->s, batch * W)) != FCH_OK) return st;
        }
        WDISPATCH_T(W, fno_pointwise, WT, grid(pts, 256), 128, s, hin, f->s, P + offset_of(f, 2, l),
                    P + offset_of(f, 3, l), f->z + l * fld, hout, batch, n2, l < f->L - 1);
    }
    WDISPATCH_T(W, fno_project, WT, grid(pts, 256), 128, s, f->h + f->L * fld, P + offset_of(f, 5, 0),
                P + offset_of(f, 6, 0), P + offset_of(f, 7, 0), P + offset_of(f, 8, 0), y, batch, n2, f->W2);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        snprintf(f->err, sizeof(f->err), "fch_fno_forward: %s", cudaGetErrorString(e));
        fch_set_thread_error(f->err);
        return FCH_ECUDA;
    }
    // keep y for the backward pass (the caller owns its array)
    e = cudaMemcpyAsync(f->y, y, (size_t)pts * 4, cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return FCH_ECUDA;
    f->a = a;
    f->have_fwd = true;
    return FCH_OK;
}

// tables and work arrays of the truncated-DFT forward pass for (B, n)
static fch_status ensure_tc(fch_fno *f, int B, int n)
{
    if (f->tc_B == B && f->tc_n == n) return FCH_OK;
    for (void *b : {(void *)f->tc_Bt, (void *)f->tc_At, (void *)f->tc_h[0], (void *)f->tc_h[1], (void *)f->tc_tw, (void *)f->tc_X, (void *)f->tc_V, (void *)f->tc_Y,
                    (void *)f->tc_Z})
        if (b) cudaFree(b);
    f->tc_Bt = f->tc_At = f->tc_h[0] = f->tc_h[1] = nullptr;
    f->tc_tw = f->tc_X = f->tc_V = f->tc_Y = f->tc_Z = nullptr;
    f->tc_B = f->tc_n = 0;
    const size_t rows = (size_t)B * f->W * n, modes = (size_t)B * f->W * f->K;
    cudaError_t e = cudaMalloc((void **)&f->tc_Bt, (size_t)32 * n * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = cudaMalloc((void **)&f->tc_At, (size_t)32 * n * sizeof(__nv_bfloat16));
    for (int i = 0; i < 2; i++)
        if (e == cudaSuccess) e = cudaMalloc((void **)&f->tc_h[i], rows * n * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = cudaMalloc((void **)&f->tc_tw, (size_t)16 * n * sizeof(float2));
    if (e == cudaSuccess) e = cudaMalloc((void **)&f->tc_X, rows * 16 * sizeof(float2));
    if (e == cudaSuccess) e = cudaMalloc((void **)&f->tc_V, rows * 16 * sizeof(float2));
    if (e == cudaSuccess) e = cudaMalloc((void **)&f->tc_Y, modes * sizeof(float2));
    if (e == cudaSuccess) e = cudaMalloc((void **)&f->tc_Z, modes * sizeof(float2));
    if (e == cudaSuccess && !f->tc_err) e = cudaMalloc((void **)&f->tc_err, sizeof(int));
    if (e == cudaSuccess) e = cudaMemsetAsync(f->tc_err, 0, sizeof(int), f->stream);
    if (e == cudaSuccess) {
        fno_dft_tables<<<grid(16L * n, 256), 256, 0, f->stream>>>(f->tc_Bt, f->tc_tw, f->tc_At, n);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        snprintf(f->err, sizeof(f->err), "fch_fno (truncated DFT): %s", cudaGetErrorString(e));
        fch_set_thread_error(f->err);
        cudaGetLastError(); // as in ensure_buffers
        return e == cudaErrorMemoryAllocation ? FCH_ENOMEM : FCH_ECUDA;
    }
    f->tc_B = B;
    f->tc_n = n;
    return FCH_OK;
}

// the forward pass with the spectral convolutions as truncated DFTs, the row DFT on
// the tensor cores (BF16 operands, FP32 sums); BF16 weights elsewhere, FP32 sums
static fch_status forward_tc(fch_fno *f, int batch, int n, const float *a, float *y)
{
    typedef __nv_bfloat16 WT;
    const WT *P = f->pbf;
    const fch_status st = ensure_tc(f, batch, n);
    if (st != FCH_OK) return st;
    const int W = f->W, M = f->M, n2 = n * n;
    const long pts = (long)batch * n2, R = (long)batch * W * n;
    cudaStream_t s = f->stream;
    {
        const WT *P0 = P + offset_of(f, 0, 0), *P1 = P + offset_of(f, 1, 0);
        const unsigned gl = grid(pts, 256);
        if (W == 16)
            fno_lift_t<WT, 16, 2><<<gl, 256, 0, s>>>(a, P0, P1, f->tc_h[0], pts, n2);
        else
            fno_lift_t<WT, 32, 2><<<gl, 256, 0, s>>>(a, P0, P1, f->tc_h[0], pts, n2);
    }
    for (int l = 0; l < f->L; l++) {
        const WT *hin = f->tc_h[l & 1];
        WT *hout = f->tc_h[(l + 1) & 1];
        const cudaError_t e = launch_rowdft_tc(hin, f->tc_Bt, f->tc_X, R, n, f->tc_err, s);
        if (e != cudaSuccess) return spec_error(f, e);
        fno_coldft<16><<<dim3(batch * W, M), 256, 2 * n * sizeof(float2), s>>>(f->tc_X, f->tc_tw + n, f->tc_Y, n);
        fno_mix_modes<WT><<<f->K, 128, (W * (W + 1) + W) * 8, s>>>(f->tc_Y, P + offset_of(f, 4, l), f->tc_Z, batch, W,
                                                                  M);
        fno_icoldft<16><<<(unsigned)((long)batch * W * (n / 64)), 256, n * sizeof(float2), s>>>(
            f->tc_Z, f->tc_tw + n, f->tc_V, (long)batch * W, n);
        // the channel mixing and the inverse x DFT: one MMA chain per 128 points
        const dim3 g((unsigned)(n / 128 * (n / kPwRows)), (unsigned)batch);
        const int act = l < f->L - 1;
        if (W == 16)
            fno_pw_tc<16><<<g, 128, 0, s>>>(hin, f->tc_V, f->tc_At, P + offset_of(f, 2, l), P + offset_of(f, 3, l),
                                           hout, n, act, f->tc_err);
        else
            fno_pw_tc<32><<<g, 128, 0, s>>>(hin, f->tc_V, f->tc_At, P + offset_of(f, 2, l), P + offset_of(f, 3, l),
                                           hout, n, act, f->tc_err);
    }
    const unsigned gp = (unsigned)(pts / 128);
    const WT *hL = f->tc_h[f->L & 1];
    if (W == 16)
        fno_proj_tc<16><<<gp, 128, 0, s>>>(hL, P + offset_of(f, 5, 0), P + offset_of(f, 6, 0), P + offset_of(f, 7, 0),
                                           P + offset_of(f, 8, 0), y, n2, f->W2, f->tc_err);
    else
        fno_proj_tc<32><<<gp, 128, 0, s>>>(hL, P + offset_of(f, 5, 0), P + offset_of(f, 6, 0), P + offset_of(f, 7, 0),
                                           P + offset_of(f, 8, 0), y, n2, f->W2, f->tc_err);
    cudaError_t e = cudaGetLastError();
    int herr = 0;
    // the tensor-core kernel's bounded waits report through a device flag
    if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, f->tc_err, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess || herr) {
        snprintf(f->err, sizeof(f->err), "fch_fno_forward (tensor cores): %s",
                 e != cudaSuccess ? cudaGetErrorString(e) : "an mbarrier wait ran out");
        fch_set_thread_error(f->err);
        return FCH_ECUDA;
    }
    f->a = a;
    f->have_fwd = true;
    return FCH_OK;
}

// refresh the bfloat16 copy of the parameters (round to nearest even)
static fch_status refresh_bf16(fch_fno *f)
{
    if (!f->pbf) return FCH_OK;
    fno_to_bf16<<<grid((long)f->np, 256), 256, 0, f->stream>>>(f->params, f->pbf, (long)f->np);
    return cudaGetLastError() == cudaSuccess ? FCH_OK : FCH_ECUDA;
}

extern "C" fch_status fch_fno_set_bf16(fch_fno *f, int on)
{
    if (!f || on < 0 || on > 2) return FCH_EINVAL;
    if (on && !f->pbf) {
        if (cudaMalloc((void **)&f->pbf, f->np * sizeof(__nv_bfloat16)) != cudaSuccess) {
            f->pbf = nullptr;
            cudaGetLastError();
            return FCH_ENOMEM;
        }
        f->tc = on == 2;
        return refresh_bf16(f);
    }
    f->tc = on == 2;
    if (!on && f->pbf) {
        cudaStreamSynchronize(f->stream);
        cudaFree(f->pbf);
        f->pbf = nullptr;
    }
    return FCH_OK;
}

extern "C" fch_status fch_fno_forward(fch_fno *f, int batch, int n, const float *a, float *y)
{
    if (!f || !a || !y || batch < 1 || n < 2 * f->M || n < 16 || n > 2048 || (n & (n - 1))) {
        fch_set_thread_error("fch_fno_forward: invalid argument");
        return FCH_EINVAL;
    }
    f->fwd_bf16 = f->pbf != nullptr;
    if (f->tc && f->pbf) {
        if (f->M != 16 || n % 128 != 0 || (f->W != 16 && f->W != 32) || f->W2 % 16 != 0) {
            fch_set_thread_error("fch_fno_forward: the tensor-core pass needs modes = 16, width 16 or 32, "
                                 "proj a multiple of 16 and n a multiple of 128");
            return FCH_EINVAL;
        }
        f->have_fwd = false;
        return forward_tc(f, batch, n, a, y);
    }
    f->have_fwd = false; // until the pass is enqueued whole: a failed one leaves nothing to go back through
    return f->pbf ? forward_impl(f, batch, n, a, y, (const __nv_bfloat16 *)f->pbf)
                  : forward_impl(f, batch, n, a, y, (const float *)f->params);
}

extern "C" fch_status fch_fno_backward(fch_fno *f, const float *target, double *loss)
{
    if (!f || !target) return FCH_EINVAL;
    if (!f->have_fwd || f->fwd_bf16) return FCH_ESTATE; // training runs on the FP32 weights
    const int B = f->B, n = f->n, W = f->W, W2 = f->W2, n2 = n * n;
    const long pts = (long)B * n2;
    const size_t fld = (size_t)B * W * n2, S = (size_t)(n / 2 + 1) * n;
    cudaStream_t s = f->stream;
    const float *P = f->params;
    float *G = f->grads;
    cudaError_t e = cudaSuccess;
    // projection and the loss (y kept by the forward pass)
    WDISPATCH(W, fno_project_bwd, grid(pts, 128), 128, s, f->h + f->L * fld, P + offset_of(f, 5, 0),
              P + offset_of(f, 6, 0), P + offset_of(f, 7, 0), f->y, target, f->dy, f->q, f->dzq, f->dh, f->sq, B,
              n2, W2, 2.0f / (float)pts);
    // partial sums in parameter order: (P, bP), (W_l, b_l) per layer, (Q1, bQ1, Q2, bQ2)
    const long oP = 0, lP = (long)W * f->cin + W, lW = (long)W * W + W, oQ = lP + f->L * lW;
    if (e == cudaSuccess) e = wgrad(f, f->dy, 1, f->q, W2, oQ + (long)W2 * W + W2);      // Q2, bQ2
    if (e == cudaSuccess) e = wgrad(f, f->dzq, W2, f->h + f->L * fld, W, oQ);            // Q1, bQ1
    for (int l = f->L - 1; l >= 0 && e == cudaSuccess; l--) {
        float *hin = f->h + l * fld;
        const float2 *R = (const float2 *)(P + offset_of(f, 4, l));
        // dz = dh act'(z); dh_l = W^T dz (into tmp)
        WDISPATCH(W, fno_pointwise_bwd, grid(pts, 128), 128, s, f->dh, f->z + l * fld, P + offset_of(f, 2, l),
                  f->dz, f->tmp, B, n2, l < f->L - 1);
        e = wgrad(f, f->dz, W, hin, W, lP + l * lW); // W_l, b_l
        if (e != cudaSuccess) break;
        // spectral branch
        if (f->modes) {
            const int BW = B * W;
            const float inv = 1.0f / ((float)n * (float)n);
            // dY = H(w(kx)/n^2 R2C(dz)); dR and the modes of the input gradient; dh = tmp +
            // C2R(n^2 v(kx) modes)
            e = field_modes(f, f->dz, f->dY, inv, 2.f * inv, 1);
            if (e == cudaSuccess) {
                fno_mode_bwd<<<f->K, 256, (W * W + 2 * BW) * 8, s>>>(f->dY, f->X + (size_t)l * BW * f->K, R,
                                                                    (float2 *)(G + offset_of(f, 4, l)), f->Ysp, BW, W);
                e = modes_field(f, f->Ysp, f->tmp, f->dh, 1.f, 0.5f);
            }
            if (e != cudaSuccess) break;
            continue;
        }
        if (fch_fft_r2c(f->plan, f->dz, f->Fd, B * W) != FCH_OK) return FCH_ECUDA;
        const int K = f->K;
        fno_dY<<<grid((long)B * W * K, 256), 256, 0, s>>>(f->Fd, f->dY, B, W, f->M, n);
        fno_dR<<<grid((long)K * W * W, 256), 256, 0, s>>>(f->dY, f->X + (size_t)l * B * W * S,
                                                          (float2 *)(G + offset_of(f, 4, l)), B, W, f->M, n);
        const int items = f->M + (f->M - 1) * (2 * f->M - 1);
        fno_dX<<<grid((long)B * W * items, 256), 256, 0, s>>>(f->dY, R, f->Ysp, B, W, f->M, n);
        if (fch_fft_c2r(f->plan, f->Ysp, f->dh, B * W) != FCH_OK) return FCH_ECUDA;
        fno_add<<<grid((long)fld, 256), 256, 0, s>>>(f->dh, f->tmp, (long)fld);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = wgrad(f, f->dh, W, f->a, f->cin, oP); // P, bP
    if (e == cudaSuccess) {
        WgRuns runs;
        runs.n = 0;
        auto run = [&](long off, long len, float *dst) {
            runs.off[runs.n] = off;
            runs.len[runs.n] = len;
            runs.dst[runs.n++] = dst;
        };
        run(oP, lP, G + offset_of(f, 0, 0));
        for (int l = 0; l < f->L; l++) run(lP + l * lW, lW, G + offset_of(f, 2, l));
        run(oQ, (long)W2 * W + 2 * W2 + 1, G + offset_of(f, 5, 0));
        int chunk;
        const int nblk = wgrad_blocks(pts, chunk);
        const long stride = (long)wgrad_stride(f);
        fno_wgrad_sum<<<grid(stride, 32), 256, 0, s>>>(f->part, nblk, stride, runs);
        e = cudaGetLastError();
    }
    // loss = mean of the squared residuals, summed in double (partials on the device)
    if (e == cudaSuccess && loss) {
        fno_loss_part<<<kLossBlocks, 256, 0, s>>>(f->sq, pts, f->lpart);
        e = cudaGetLastError();
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(f->hsum, f->lpart, kLossBlocks * sizeof(double), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        double acc = 0;
        for (int i = 0; i < kLossBlocks; i++) acc += f->hsum[i];
        if (e == cudaSuccess) *loss = acc / (double)pts;
    }
    if (e != cudaSuccess) {
        snprintf(f->err, sizeof(f->err), "fch_fno_backward: %s", cudaGetErrorString(e));
        fch_set_thread_error(f->err);
        return FCH_ECUDA;
    }
    return FCH_OK;
}

extern "C" fch_status fch_fno_adam(fch_fno *f, float lr, float beta1, float beta2, float eps)
{
    if (!f || !(lr > 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) || !(eps > 0)) return FCH_EINVAL;
    f->adam_t++;
    const float c1 = 1.f - powf(beta1, (float)f->adam_t), c2 = 1.f - powf(beta2, (float)f->adam_t);
    fno_adam<<<grid((long)f->np, 256), 256, 0, f->stream>>>(f->params, f->grads, f->am, f->av, (long)f->np, lr, beta1,
                                                            beta2, eps, c1, c2);
    if (cudaGetLastError() != cudaSuccess) return FCH_ECUDA;
    return refresh_bf16(f);
}

__global__ void fno_gelu_eval(const float *__restrict__ x, float *__restrict__ y, long cnt, int as)
{
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (!as) {
        if (t < cnt) y[t] = gelu(x[t]);
        return;
    }
    // the inference GELU works on pairs: elements 2t and 2t + 1 (the last alone twice)
    const long i = 2 * t;
    if (i >= cnt) return;
    const bool pair = i + 1 < cnt;
    const float2 g = x2_split(gelu_as2(x2(x[i], pair ? x[i + 1] : x[i])));
    y[i] = g.x;
    if (pair) y[i + 1] = g.y;
}

// test hook (not part of the C ABI of fch.h): the GELU of the inference kernels
// (as = 1) or of the training path (as = 0) on cnt device floats; 0 or a status
extern "C" int fch_debug_fno_gelu(const float *x, float *y, long cnt, int as, void *stream)
{
    if (!x || !y || cnt < 1) return FCH_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    fno_gelu_eval<<<grid(cnt, 256), 256, 0, s>>>(x, y, cnt, as);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        fch_set_thread_error(cudaGetErrorString(e));
        return FCH_ECUDA;
    }
    return FCH_OK;
}

// test hook (not part of the C ABI of fch.h): the tensor-core row DFT alone,
// X[r][kx] for kx < 16 of R rows of n floats (device arrays); returns 0 or a status
extern "C" int fch_debug_rowdft_tc(const float *h, float *X, int R, int n, void *stream)
{
    if (!h || !X || R < 1 || n < 64 || n % 64 != 0 || n > 2048) return FCH_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    __nv_bfloat16 *Bt = nullptr, *hb = nullptr;
    float2 *tw = nullptr;
    int *err = nullptr, herr = 0;
    cudaError_t e = cudaMalloc((void **)&Bt, (size_t)32 * n * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = cudaMalloc((void **)&tw, (size_t)16 * n * sizeof(float2));
    if (e == cudaSuccess) e = cudaMalloc((void **)&err, sizeof(int));
    if (e == cudaSuccess) e = cudaMemsetAsync(err, 0, sizeof(int), s);
    if (e == cudaSuccess) e = cudaMalloc((void **)&hb, (size_t)R * n * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) {
        fno_dft_tables<<<grid(16L * n, 256), 256, 0, s>>>(Bt, tw, nullptr, n);
        fno_to_bf16<<<grid((long)R * n, 256), 256, 0, s>>>(h, hb, (long)R * n);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = launch_rowdft_tc(hb, Bt, (float2 *)X, R, n, err, s);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    for (void *b : {(void *)Bt, (void *)hb, (void *)tw, (void *)err})
        if (b) cudaFree(b);
    if (e != cudaSuccess) {
        fch_set_thread_error(cudaGetErrorString(e));
        return FCH_ECUDA;
    }
    return herr ? FCH_ECUDA : FCH_OK;
}
