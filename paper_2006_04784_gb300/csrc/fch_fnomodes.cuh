// fch_fnomodes.cuh -- the FNO's spectral branch in single precision on grids up to 256^2:
// a field's transform to its retained modes, and back, by one block without the full
// spectrum ever leaving it, and the products over the modes one block a mode.
//
// A block transforms one field of n x n: the rows two at a time (row 2j + i row 2j + 1 as
// one complex sequence, n / 8 threads each, fft_reg of the stepping passes), the M retained
// kx of each kept in shared memory (M columns of n), then those columns along y; out go the
// M (2M - 1) retained modes. The inverse runs backwards. The plans' transforms moved every
// field's full half spectrum through memory twice each way for 496 of its 8320 modes (128^2,
// M = 16: sixteen transforms of 256 fields took 0.6 of a 1.49 ms training step).
//
// Modes are stored mode-major, [kx (2M-1) + kyi][field], so that a mode's products over the
// channels read and write contiguous vectors; weights [m][o][i] are read as they lie. (The
// products before ran over modes in the fastest index, weights 8 KB apart between lanes.)
#pragma once
#include "fch_reg.cuh"

namespace fch {

// threads and shared memory of the field transforms; columns are padded to whole warps
template <int LOGN> struct FnoModes {
    static constexpr int n = 1 << LOGN, tps = n / 8, SL = n + n / 8;
    static constexpr int threads = n * n / 16 < 256 ? n * n / 16 : 256;
    static constexpr int groups = threads / tps; // sequences transformed at once
    static constexpr int per_warp = 32 / tps;
    __host__ __device__ static constexpr int cols(int M) { return (M + per_warp - 1) / per_warp * per_warp; }
    __host__ __device__ static constexpr int smem(int M)
    {
        return (groups * SL + cols(M) * SL + M * (2 * M - 1)) * 8;
    }
};

__device__ __forceinline__ int fno_ky(int q, int M, int n) { return q < M ? q : n - (q - M + 1); }

// out[m][field] = s(kx) F(m) of field blockIdx.x, F its R2C, s = s0 at kx = 0 (through its
// Hermitian part when herm), else s1
template <int LOGN>
__global__ void __launch_bounds__(FnoModes<LOGN>::threads)
fno_field_modes(const float *__restrict__ h, float2 *__restrict__ out, const float2 *__restrict__ tw, int M,
                float s0, float s1, int herm)
{
    typedef FnoModes<LOGN> G;
    constexpr int n = G::n, TPS = G::tps, SL = G::SL;
    extern __shared__ __align__(16) float2 fm_smem[];
    const int g = threadIdx.x / TPS, t = threadIdx.x % TPS;
    float2 *buf = fm_smem + g * SL, *cols = fm_smem + G::groups * SL, *none = nullptr;
    const float *f = h + (long)blockIdx.x * n * n + t;
    float2 v[8];
#pragma unroll 1
    for (int j = g; j < n / 2; j += G::groups) { // whole warps: groups divides n / 2
#pragma unroll
        for (int m = 0; m < 8; m++) v[m].x = f[(2 * j) * n + TPS * m];
#pragma unroll
        for (int m = 0; m < 8; m++) v[m].y = f[(2 * j + 1) * n + TPS * m];
        fft_reg<LOGN, 8, false, true>(v, buf, none, tw, t);
        __syncwarp();
#pragma unroll
        for (int m = 0; m < 8; m++) buf[skew(t + TPS * m)] = v[m];
        __syncwarp();
        for (int kx = t; kx < M; kx += TPS) {
            const float2 z0 = buf[skew(kx)], z1 = buf[skew((n - kx) & (n - 1))];
            // row 2j: (z0 + conj z1) / 2, row 2j + 1: (z0 - conj z1) / (2i)
            cols[kx * SL + skew(2 * j)] = make_float2(0.5f * (z0.x + z1.x), 0.5f * (z0.y - z1.y));
            cols[kx * SL + skew(2 * j + 1)] = make_float2(0.5f * (z0.y + z1.y), 0.5f * (z1.x - z0.x));
        }
        __syncwarp();
    }
    __syncthreads();
    const int K2 = 2 * M - 1, nc = G::cols(M);
#pragma unroll 1
    for (int kx = g; kx < nc; kx += G::groups) { // nc is whole warps of sequences
        float2 *c = cols + kx * SL;
#pragma unroll
        for (int m = 0; m < 8; m++) v[m] = kx < M ? c[skew(t + TPS * m)] : make_float2(0.f, 0.f);
        fft_reg<LOGN, 8, false, true>(v, buf, none, tw, t);
#pragma unroll
        for (int m = 0; m < 8; m++) c[skew(t + TPS * m)] = v[m];
        __syncwarp();
        if (kx < M) {
            const float s = kx ? s1 : s0;
            for (int q = t; q < K2; q += TPS) {
                const int ky = fno_ky(q, M, n);
                float2 z = c[skew(ky)];
                if (herm && kx == 0) {
                    const float2 w = c[skew((n - ky) & (n - 1))];
                    z = make_float2(0.5f * (z.x + w.x), 0.5f * (z.y - w.y));
                }
                out[(long)(kx * K2 + q) * gridDim.x + blockIdx.x] = make_float2(s * z.x, s * z.y);
            }
        }
    }
}

// out (+)= the real field of the modes s(kx) Y[m][field]: C2R without its 1/n^2, the kx = 0
// modes through their Hermitian part. add: out = base + field, else out = field.
template <int LOGN>
__global__ void __launch_bounds__(FnoModes<LOGN>::threads)
fno_modes_field(const float2 *__restrict__ Y, const float *__restrict__ base, float *__restrict__ out,
                const float2 *__restrict__ tw, int M, float s0, float s1)
{
    typedef FnoModes<LOGN> G;
    constexpr int n = G::n, TPS = G::tps, SL = G::SL;
    extern __shared__ __align__(16) float2 fm_smem[];
    const int g = threadIdx.x / TPS, t = threadIdx.x % TPS;
    float2 *buf = fm_smem + g * SL, *cols = fm_smem + G::groups * SL, *none = nullptr;
    const int K2 = 2 * M - 1, nc = G::cols(M);
    float2 *ym = cols + nc * SL;
    for (int m = threadIdx.x; m < M * K2; m += G::threads) ym[m] = Y[(long)m * gridDim.x + blockIdx.x];
    __syncthreads();
    float2 v[8];
#pragma unroll 1
    for (int kx = g; kx < nc; kx += G::groups) {
        const float s = kx ? s1 : s0;
#pragma unroll
        for (int m = 0; m < 8; m++) {
            const int ky = t + TPS * m;
            const int q = ky < M ? ky : ky > n - M ? n - ky + M - 1 : -1;
            float2 z = make_float2(0.f, 0.f);
            if (kx < M && q >= 0) {
                z = ym[kx * K2 + q];
                if (kx == 0) { // (Y(ky) + conj Y(-ky)) / 2
                    const float2 w = ym[ky == 0 ? 0 : ky < M ? ky + M - 1 : n - ky];
                    z = make_float2(0.5f * (z.x + w.x), 0.5f * (z.y - w.y));
                }
            }
            v[m] = make_float2(s * z.x, -s * z.y); // the inverse as conj, forward, conj
        }
        fft_reg<LOGN, 8, false, true>(v, buf, none, tw, t);
#pragma unroll
        for (int m = 0; m < 8; m++) cols[kx * SL + skew(t + TPS * m)] = make_float2(v[m].x, -v[m].y);
    }
    __syncthreads();
    const long f0 = (long)blockIdx.x * n * n + t;
#pragma unroll 1
    for (int j = g; j < n / 2; j += G::groups) {
#pragma unroll
        for (int m = 0; m < 8; m++) {
            const int k = t + TPS * m, kk = k < M ? k : n - k;
            float2 z = make_float2(0.f, 0.f);
            if (kk < M) {
                // row 2j + i row 2j + 1 at k; at n - k the conjugates of both
                const float2 a = cols[kk * SL + skew(2 * j)], b = cols[kk * SL + skew(2 * j + 1)];
                if (k == 0)
                    z = make_float2(a.x, b.x);
                else if (k < M)
                    z = make_float2(a.x - b.y, a.y + b.x);
                else
                    z = make_float2(a.x + b.y, b.x - a.y);
            }
            v[m] = make_float2(z.x, -z.y);
        }
        fft_reg<LOGN, 8, false, true>(v, buf, none, tw, t);
#pragma unroll
        for (int m = 0; m < 8; m++) {
            const long a = f0 + (2 * j) * n + TPS * m;
            out[a] = base ? base[a] + v[m].x : v[m].x;
            out[a + n] = base ? base[a + n] - v[m].y : -v[m].y;
        }
    }
}

} // namespace fch
