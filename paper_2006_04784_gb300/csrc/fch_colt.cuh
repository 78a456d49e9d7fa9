// fch_colt.cuh -- column passes of the standalone single-precision transforms at
// N = 1024 with their input staged by the TMA engine.
//
// A tile is P = 2 column pairs: four columns, 32 bytes of every row of the
// pair-layout work array Z. 512 threads: thread (c, t) = (tid mod 4, tid / 4) holds the
// points t + 128 m of column c at both ends of the transform, as the passes built for a
// size do (fch_reg.cuh: column N - kx in its conjugate, inverses as conj, forward, conj).
// Blocks are persistent: block b takes tiles b, b + B, b + 2B, ... of all the launch's field
// pairs (tile g: pair g / 256, column pairs 2 (g mod 256) and the next), and the next tile's
// input lands in a 32 KB stage while the current tile is transformed:
//  - forward (R2C): four 2D tensor-map boxes of Z (256 rows x 8 floats each,
//    cp.async.bulk.tensor) fill the stage densely, row n at 32 n bytes; a warp's reads of
//    the first stage's inputs are 256 contiguous bytes;
//  - inverse (C2R): the rows kx of the two half spectra (8 KB each, cp.async.bulk) of the
//    tile's two column pairs; both columns of a pair read the same index, natural order.
//    The tile of pair 0 (kx = 0 and N/2 need four rows) reads its spectra from global memory.
// The Hermitian split of the forward pass trades one value of a work item each way between
// lanes c = 0, 1 (2, 3) by shuffles; the inverse stores straight from the last stage, whole
// 32-byte sectors. Shared memory carries the three exchanges between the stages only: the
// kernel before went through it eight times a transform (MIO throttle its first stall) and
// took 38.4 us forward, 50.1 us inverse for eight field pairs.
// Copies complete in bytes on the block's mbarrier; a wait that runs out of time (1 s)
// sets *kp.err, and the block stops after waiting (bounded) for the copy it started.
#pragma once
#include <cuda.h>
#include "fch_reg.cuh"
#include "fch_tc.cuh"

namespace fch {

constexpr int kColtThreads = 512;
constexpr int kColtStageBytes = 4 * 1024 * 8;           // the next tile's input
constexpr int kColtSC = 1152 + 4;                       // a skewed column; the four start 4 elements apart mod 16
constexpr int kColtTileBytes = 4 * kColtSC * 8;
constexpr int kColtTwBytes = 1024 * 8;                  // the per-stage twiddles, loaded once a block
constexpr int kColtSmem = kColtStageBytes + kColtTileBytes + kColtTwBytes + 16 + 128; // + mbarrier, + slack
constexpr uint64_t kColtWaitNs = 1000000000ull;

template <int MODE>
__global__ void __launch_bounds__(kColtThreads, 2) col_pass_t(const fch_kparams kp,
                                                              const __grid_constant__ CUtensorMap zmap)
{
    static_assert(MODE == CM_FWD_STORE || MODE == CM_INV_LOAD, "the standalone transform modes");
    typedef float2 C;
    constexpr bool FWD = MODE == CM_FWD_STORE;
    constexpr int N = 1024, NC = 4, NT = kColtThreads, H = 4;
    pdl_begin();
    extern __shared__ unsigned char smem_raw[];
    // the TMA destination wants 128-byte alignment
    unsigned char *base = smem_raw + ((128u - (fch::tc::smem_u32(smem_raw) & 127u)) & 127u);
    C *stage = (C *)base;
    C *tile = (C *)(base + kColtStageBytes);
    C *tw = (C *)(base + kColtStageBytes + kColtTileBytes);
    uint64_t *bar = (uint64_t *)(base + kColtStageBytes + kColtTileBytes + kColtTwBytes);
    const int c = threadIdx.x % NC, t = threadIdx.x / NC, side = c & 1, pp = c >> 1;
    const long npairs = kp.npairs > 1 ? kp.npairs : 1;
    const long ntiles = npairs * (N / 4);
    for (int i = threadIdx.x; i < N; i += NT) tw[i] = ldg((const C *)kp.tw + i);
    const float inv_n2 = kp.cf.inv_n2;
    const bool two = kp.in1 != nullptr; // inverse: a second half spectrum

    // a tile's input reaches the stage unless it is an inverse tile of pair 0
    auto staged = [&](long g) { return FWD || (g & 255) != 0; };
    auto fetch = [&](long g) { // thread 0
        const long pr = g >> 8;
        const int p0 = 2 * (int)(g & 255);
        if (FWD) {
            fch::tc::mbar_expect_tx(bar, kColtStageBytes);
#pragma unroll
            for (int q = 0; q < 4; q++)
                fch::tc::tma_load_2d(stage + q * 256 * NC, &zmap, 4 * p0, (int)(pr * N + 256 * q), bar);
        } else if (p0 != 0) {
            const char *i0 = (const char *)kp.in0 + pr * kp.pstride_in;
            const char *i1 = two ? (const char *)kp.in1 + pr * kp.pstride_in : nullptr;
            fch::tc::mbar_expect_tx(bar, (two ? 4 : 2) * N * 8);
#pragma unroll
            for (int q = 0; q < 2; q++) {
                fch::tc::bulk_g2s(stage + 2 * q * N, i0 + (long)(p0 + q) * N * 8, N * 8, bar);
                if (two) fch::tc::bulk_g2s(stage + (2 * q + 1) * N, i1 + (long)(p0 + q) * N * 8, N * 8, bar);
            }
        }
    };

    long g = blockIdx.x;
    if (threadIdx.x == 0) {
        fch::tc::mbar_init(bar, 1);
        fch::tc::mbar_init_fence();
        if (g < ntiles) fetch(g);
    }
    __syncthreads();
    uint32_t phase = 0;
    bool ok = true;
    for (; g < ntiles; g += gridDim.x) {
        const long pr = g >> 8;
        const int p0 = 2 * (int)(g & 255), p = p0 + pp;
        if (staged(g)) {
            ok = __syncthreads_and(fch::tc::mbar_wait(bar, phase, kColtWaitNs));
            if (!ok) break;
            phase ^= 1u;
        }
        C v[8];
        if (FWD) {
            const unsigned m1 = side ? 0x80000000u : 0u;
#pragma unroll
            for (int m = 0; m < 8; m++) {
                v[m] = stage[(t + 128 * m) * NC + c];
                v[m].y = flip(v[m].y, m1);
            }
        } else {
            // (C, D) the two half spectra over N^2: column kx holds conj(C + i D), column
            // N - kx C* + i D* at the same index (pair 0: column N/2 holds C + i D of -k)
            const bool own = p0 == 0 && pp == 0;
            const C *a, *b;
            if (staged(g)) {
                a = stage + 2 * pp * N;
                b = stage + (2 * pp + 1) * N;
            } else {
                const long kx = own ? (side ? N / 2 : 0) : 1;
                a = (const C *)((const char *)kp.in0 + pr * kp.pstride_in) + kx * N;
                b = two ? (const C *)((const char *)kp.in1 + pr * kp.pstride_in) + kx * N : a;
            }
#pragma unroll
            for (int m = 0; m < 8; m++) {
                const int k = t + 128 * m, kk = own && side ? (N - k) & (N - 1) : k;
                const C Co = cscale(a[kk], inv_n2);
                const C Do = two ? cscale(b[kk], inv_n2) : mk<C>(0.f, 0.f);
                if (!side)
                    v[m] = mk<C>(Co.x - Do.y, -(Co.y + Do.x));
                else if (!own)
                    v[m] = mk<C>(Co.x + Do.y, Do.x - Co.y);
                else
                    v[m] = mk<C>(Co.x - Do.y, Co.y + Do.x);
            }
        }
        C *buf = tile + c * kColtSC, *none = nullptr;
        reg_stage<10, 8, 3, 0, false, false, false>(v, buf, none, (const C *)tw, t);
        // the exchange's barriers: every thread has read the stage
        if (threadIdx.x == 0) {
            fch::tc::fence_async_smem(); // the stage's reads come before the next copy's writes
            if (g + gridDim.x < ntiles) fetch(g + gridDim.x);
        }
        reg_stage<10, 8, 3, 1, false, false, false>(v, buf, none, (const C *)tw, t);
        reg_stage<10, 8, 3, 2, false, false, false>(v, buf, none, (const C *)tw, t);
        reg_stage<10, 8, 1, 3, false, false, false>(v, buf, none, (const C *)tw, t);
        if (FWD) {
            C *o0 = (C *)((char *)kp.out0 + pr * kp.pstride_out);
            C *o1 = kp.out1 ? (C *)((char *)kp.out1 + pr * kp.pstride_out) : nullptr;
            // A = (za + zb) / 2, B = (za - zb) / (2i), za = Z(kx, ky), zb = conj Z(N - kx, -ky)
            auto split = [&](C za, C zb, long idx) {
                o0[idx] = cscale(cadd(za, zb), 0.5f);
                if (o1) {
                    const C dm = csub(za, zb);
                    o1[idx] = mk<C>(0.5f * dm.y, -0.5f * dm.x);
                }
            };
            C r[H]; // the partner column's values of this thread's work items
#pragma unroll
            for (int i = 0; i < H; i++) {
                const C s = side ? v[i] : v[i + H];
                r[i] = mk<C>(__shfl_xor_sync(0xffffffffu, s.x, 1), __shfl_xor_sync(0xffffffffu, s.y, 1));
            }
            if (p0 == 0) { // pair 0: columns 0 and N/2 pair row k with row -k of themselves
#pragma unroll
                for (int m = 0; m < 8; m++) buf[skew(t + 128 * m)] = v[m];
                __syncthreads();
            }
            if (p > 0) {
#pragma unroll
                for (int i = 0; i < H; i++) {
                    const int ky = t + 128 * (side ? i + H : i);
                    split(side ? r[i] : v[i], side ? v[i + H] : r[i], (long)p * N + ky);
                }
            } else {
#pragma unroll
                for (int m = 0; m < 8; m++) {
                    const int k = t + 128 * m, km = (N - k) & (N - 1);
                    const C zm = buf[skew(km)];
                    split(side ? cconj(v[m]) : v[m], side ? zm : cconj(zm), side ? (long)(N / 2) * N + km : k);
                }
            }
            if (p0 == 0) __syncthreads(); // the tile is read before the next tile's first writes
        } else {
            const unsigned m0 = side ? 0u : 0x80000000u;
            C *Z = (C *)kp.Z + pr * N * N + 2 * p0 + c;
#pragma unroll
            for (int m = 0; m < 8; m++) {
                v[m].y = flip(v[m].y, m0);
                __stcg(Z + (long)(t + 128 * m) * N, v[m]);
            }
        }
    }
    if (!ok && threadIdx.x == 0) {
        // the copy this block waits for may still land: let it, then report
        fch::tc::mbar_wait(bar, phase, kColtWaitNs);
        if (kp.err) atomicExch(kp.err, 1);
    }
}

} // namespace fch
