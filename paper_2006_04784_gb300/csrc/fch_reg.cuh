// fch_reg.cuh -- the row and column passes built for a grid size, with the ends of the
// transforms in registers.
//
// A sequence of N = 2^LOGN points belongs to tps = N / PPT threads; thread t holds the
// points t + tps m, m < PPT ("natural" slots), before the first and after the last
// Stockham stage: the first stage's butterflies read exactly those points, and the last
// stage's write exactly those. So the passes load the work array straight into the first
// stage, run the pointwise or spectral stage on the registers the last stage leaves, hand
// them to the first stage of the transform back, and store from its last stage: shared
// memory carries only the exchanges between stages (one store and one load a point per
// exchange, one stage fewer than the transform has), where the shared-memory kernels
// (row_pass, col_pass) go through it at both ends of every stage with two barriers each.
//
// Inverse transforms run as conj, forward, conj, with the transform's code in a loop over
// the two directions: one copy of the (long, unrolled) butterfly code a kernel, since a
// small grid's pass runs its code once or twice a warp and waits for instructions.
//
// Column pass: the pair (kx, N - kx) is transformed with column N - kx conjugated on
// load. Its transform at index ky is then conj Z(N - kx, -ky), the partner the Hermitian
// split of (kx, ky) needs, at the same thread and register as Z(kx, ky): the two threads
// of a work item trade one value each way through shared memory at their own natural
// slots (lanes c = 0, 1 of the same warp, or the two blocks of a cluster).
#pragma once
#include <type_traits>
#include "fch_kernels.cuh"

namespace fch {

// x or -x by flipping the sign bits with mask (0 or 0x80000000): no FP64 operation
__device__ __forceinline__ float flip(float x, unsigned m) { return __uint_as_float(__float_as_uint(x) ^ m); }
__device__ __forceinline__ double flip(double x, unsigned m)
{
    return __hiloint2double(__double2hiint(x) ^ (int)m, __double2loint(x));
}
__device__ __forceinline__ df flip(df x, unsigned m) { return df(flip(x.hi, m), flip(x.lo, m)); }

// the passes standalone transforms run
constexpr bool row_xf(int mode) { return mode == RM_R2C_LOAD || mode == RM_C2R_STORE; }
constexpr bool col_xf(int mode) { return mode == CM_FWD_STORE || mode == CM_INV_LOAD; }

// What a pass is built for, by element (16 bytes: double and double-float; 8: single) and
// size. Points a thread: two (radix-8 stages level by level) where a pass is a few warps on
// the 608 sub-partitions and the time is the dependent chain of one of them, in double to
// 128^2 and in the others to 256^2; four (radix-4) in double at 256^2, in double-float to 1024^2 and
// in single at 512^2; eight (radix-8 stages, fewer exchanges and twiddle products) where
// the pipes are the bound or the blocks would get too large. Two points cost as many
// operations as four (22 a point of a 128-point transform) and twice the exchanges, but
// halve the instructions of a warp, and a double-precision one holds its sub-partition for
// 64 cycles whatever its lanes do. Blocks an SM: enough registers that nothing spills; at
// 1024^2 four blocks of 256 threads (two waves whose loads, transforms and stores overlap)
// beat seven of 128 in one wave, whose phases run in step.
// Adaptive IMEX passes, GB300, us a run of the case: double-float 1024^2, 48 trials: 8
// points x 7 blocks 6346, x 5 6313, 4 points x 3 6484, x 4 6198, two buffers 6133;
// 2048^2, 32 trials: 8 points 14.4k, 4 points 17.0k; 512^2, 24 trials: 4 points 1125, 2
// points 1280; 256^2, 64 trials: 4 points 1984, 2 points 1726, PSD 2573, 2345 (in a sweep
// with 512^2 and 1024^2 grids, which fill the GPU, 2 points lose 1.7 %: 8073, 8210; six 256^2
// grids alone gain: 1844, 1578); 128^2, 24 trials: 749, 602, PSD 2101, 1718. Double
// 1024^2, 12 trials: 8 points x 5 7426, x 7 7568, 4 points x 4 7632; 512^2 SAV, 32 trials: 8
// points 6424, 4 points 6672; 256^2 PSD, 24 trials: 4 points 4703, 2 points 4826; 128^2, 100
// fixed steps: 8 points 5430, 4 points 2946 (with what came between), 2 points 2111. Single, 50 fixed IMEX steps: 128^2 8 points 767, 4 points 606, 2
// points 557; 256^2 760, 664, 658; 512^2 SAV, 24 steps: 761, 695, 747.
// Transforms on their own (XF) run many fields at once: eight points in single at all sizes
// (33 fields of 256^2 there and back 31.6 us, 4 points 32.6, 2 points 43.1); in double as
// the steps (128^2, one pair 19.7 -> 14.6 us at 2 points, 8 pairs 33.3 -> 35.1, 16 pairs and
// an odd field 77.8 -> 73.8). One choice for every batch: a field's result does not depend
// on how many are transformed with it.
template <typename T> constexpr int reg_points(int logn, bool xf)
{
    return sizeof(T) == 4                  ? (xf ? 8 : logn <= 8 ? 2 : logn == 9 ? 4 : 8)
           : std::is_same<T, df>::value ? (logn <= 8 ? 2 : logn <= 10 ? 4 : 8)
                                           : (logn <= 7 ? 2 : logn <= 8 ? 4 : 8);
}

// points a thread of the built pass that a launch takes, 0 where it takes another kernel: tile
// 0, N = 64 ... 2048, and the twiddle table that the pass reads at hand (the radix-4 one is
// kept by contexts and plans, not by fch_fft_r2c_noalloc)
template <typename T> inline int reg_pass(const fch_kparams &kp, int tile, bool xf)
{
    if (tile != 0 || kp.logN < 6 || kp.logN > 11) return 0;
    const int p = reg_points<T>(kp.logN, xf);
    return (p == 4 ? kp.tw4 : kp.tw) ? p : 0;
}

template <typename T, int LOGN, bool XF> struct RegCfg {
    static constexpr bool single = sizeof(T) == 4, dfl = std::is_same<T, df>::value;
    static constexpr int N = 1 << LOGN;
    static constexpr int ppt = reg_points<T>(LOGN, XF);
    static constexpr int tps = N / ppt;
    // rows: whole warps
    static constexpr int rpb = tps >= 32 ? 1 : 32 / tps;
    static constexpr int row_threads = rpb * tps;
    static constexpr int row_minb = LOGN == 10 ? (dfl ? 4 : single ? 8 : 5) : LOGN == 11 ? 3 : LOGN == 9 ? 4 : 1;
    // columns: P pairs a block; at N = 1024 in 16-byte elements a cluster of two blocks, one
    // column each (1024 blocks fill the 152 SMs evenly where 512 leave a sixth idle)
    static constexpr bool cl = !single && LOGN == 10;
    static constexpr int P = single ? 2 : 1;
    static constexpr int ncol = cl ? 1 : 2 * P;
    static constexpr int col_threads = ncol * tps;
    static constexpr int col_blocks = cl ? N : N / (2 * P);
    static constexpr int col_minb = cl ? (dfl ? 4 : 5) : LOGN == 11 ? (single ? 1 : 2) : LOGN == 9 && !single ? 2 : 1;
    // programmatic launch: the successor may start launching at once where the passes fill
    // the GPU (its blocks can only take slots that free up), when the block stores its
    // results elsewhere (blocks waiting on idle SMs crowd the running pass: at 256^2 an
    // early start costs 4 %, a late one saves 7 %)
    static constexpr bool early = LOGN >= 10;
    // large grids: a prefetch of the spectra's rows, and work items in flight at once
    static constexpr bool prefetch = LOGN >= 10;
    static constexpr int items = LOGN == 10 && dfl ? 2 : 1;
    // shared memory: one sequence skewed; two buffers alternate where they fit easily
    // (one barrier an exchange), one elsewhere (two barriers)
    static constexpr bool db = LOGN <= 9 || (LOGN == 10 && dfl);
    static constexpr int SL = N + N / 8;
    // columns of a block interleave over the lanes: their buffers start 4 elements apart
    // modulo 16, so that the lanes of one access fall on distinct banks
    static constexpr int SC = cl ? SL : (SL + 15) / 16 * 16 + 4;
    static constexpr int csz = single ? 8 : 16;
    static constexpr int row_smem = (db ? 2 : 1) * rpb * SL * csz;
    static constexpr int col_smem = (db ? 2 : 1) * ncol * SC * csz;
};

// Forward transform of the natural slots v (in and out). buf: the sequence's buffer (the
// exchanges alternate with buf2 when DB); on return buf is the one the next exchange may
// write first. WS: the sequence's threads lie in one warp.
template <bool WS> __device__ __forceinline__ void seq_sync()
{
    if (WS)
        __syncwarp();
    else
        __syncthreads();
}

// A stage of radix R = 2^LR and sub-length Ns = 8^S by threads of two points. Its butterflies
// run level by level in the order of eight points a thread (bfly8: the same products and
// sums, twiddles from the table of radix-8 stages), the threads (j, c) = (t mod N/R, t / (N/R))
// of butterfly j trading values between the levels through the natural slots j + (N/R) q:
// level 1 takes the points c and c + R/2, level 2 the sums (c even) or differences (c odd) of
// the even (c < 2) or odd points, level 3 the outputs k = c of both halves. (Radix-2 stages
// with a twiddle product each cost as many instructions and exchanges and take the same time,
// but round more. F(u) in single precision at 64^2, q = 0.5: 1.16e-4 from 64 bits, as here
// 1.08e-4; a double transform of noise at 64^2: 3.16e-16, here 2.70e-16.)
// Double-float is renormalised at the end of every stage: F(u) at 256^2, q = 0, 8.9e-13 from
// 64 bits, after the first and last 1.03e-12, after the last alone 1.27e-12 (radix-2 stages
// 1.09e-12); 64 IMEX trials 1723, 1721, 1722 us.
// The twiddles of all stages are read before the first: read in their stages, the first
// point's in a branch, the same trials take 1838 us.
template <bool DB, bool WS, typename C>
__device__ __forceinline__ void reg_trade2(C *v, C *&buf, C *&buf2, int w0, int w1, int t, int half)
{
    if (!DB) seq_sync<WS>();
    buf[skew(w0)] = v[0];
    buf[skew(w1)] = v[1];
    seq_sync<WS>();
    v[0] = buf[skew(t)];
    v[1] = buf[skew(t + half)];
    if (DB) {
        C *o = buf;
        buf = buf2;
        buf2 = o;
    }
}
// the twiddles of a stage's two points (the first where c > 0), read before the transform
template <int LOGN, int LR, int S, typename C>
__device__ __forceinline__ void reg_twiddles2(C *w, const C *__restrict__ tw, int t)
{
    constexpr int LB = LOGN - LR, Ns = 1 << (3 * S);
    const int c = t >> LB;
    tw += (Ns - 8) + (t & ((1 << LB) - 1) & (Ns - 1));
    w[0] = ldg(tw + (c > 0 ? c - 1 : 0) * Ns);
    w[1] = ldg(tw + (c + (1 << LR >> 1) - 1) * Ns);
}
template <int LOGN, int LR, int S, bool DB, bool WS, typename C>
__device__ __forceinline__ void reg_stage2(C *v, C *&buf, C *&buf2, const C *w, int t)
{
    typedef decltype(C().x) R;
    constexpr int N = 1 << LOGN, LB = LOGN - LR, NB = 1 << LB, Ns = 1 << (3 * S);
    constexpr bool last = (Ns << LR) == N;
    static_assert(LR == 3 || last, "stages of radix 2 and 4 come last");
    const int j = t & (NB - 1), c = t >> LB;
    if (Ns > 1) {
        if (c > 0) v[0] = btw(v[0], w[0]);
        v[1] = btw(v[1], w[1]);
    }
    bfly2<-1>(v[0], v[1]);
    if (LR >= 2) {
        const int q = LR == 3 ? 2 * (c & 1) + 4 * (c >> 1) : 2 * c;
        reg_trade2<DB, WS>(v, buf, buf2, j + q * NB, j + (q + 1) * NB, t, N / 2);
        if (c & 1) v[1] = mk<C>(v[1].y, flip(v[1].x, 0x80000000u));
        bfly2<-1>(v[0], v[1]);
    }
    if (LR == 3) {
        const int q = (c & 1) + 4 * (c >> 1);
        reg_trade2<DB, WS>(v, buf, buf2, j + q * NB, j + (q + 2) * NB, t, N / 2);
        const C e = v[0];
        C o = v[1];
        if (c & 2) o = mk<C>(o.y, flip(o.x, 0x80000000u));
        const R s = (R)0.70710678118654752440;
        if (NB >= 32) { // whole warps of one c
            if (c & 1) {
                bscaled(e, mk<C>(radd(o.x, o.y), rsub(o.y, o.x)), s, v[0], v[1]);
            } else {
                v[0] = badd(e, o);
                v[1] = bsub(e, o);
            }
        } else {
            const C x = mk<C>(radd(o.x, o.y), rsub(o.y, o.x));
            bscaled(e, c & 1 ? x : o, c & 1 ? s : (R)1, v[0], v[1]);
        }
    }
    v[0] = bnorm(v[0]);
    v[1] = bnorm(v[1]);
    if (!last) {
        const int d = ((j >> (3 * S)) << (3 * S + LR)) + (j & (Ns - 1)) + c * Ns;
        reg_trade2<DB, WS>(v, buf, buf2, d, d + 4 * Ns, t, N / 2);
    }
}

// Radix-4 stages renormalise double-float after the third as well as at the end, their
// rounding being that of more stages than radix 8 has: F(u) at 512^2, q = 0, 1.14e-12 from 64
// bits, without 1.45e-12 (eight points 1.39e-12), at 1024^2 1.21e-12, 1.57e-12 (1.54e-12);
// 48 IMEX trials of 1024^2 6007 -> 6058 us.
// (TWG: the twiddles lie in global memory, read through the read-only cache; else shared)
template <int LOGN, int PPT, int LR, int S, bool DB, bool WS, bool TWG = true, typename C>
__device__ __forceinline__ void reg_stage(C *v, C *&buf, C *&buf2, const C *__restrict__ tw, int t)
{
    constexpr int N = 1 << LOGN, tps = N / PPT, LP = PPT == 8 ? 3 : 2;
    constexpr int R = 1 << LR, NB = PPT / R;
    constexpr int lNs = S * LP, Ns = 1 << lNs;
    constexpr bool last = (Ns << LR) == N;
#pragma unroll
    for (int b = 0; b < NB; b++) {
        const int j = t + b * tps;
        C x[R];
#pragma unroll
        for (int r = 0; r < R; r++) x[r] = v[b + NB * r];
        if (Ns > 1) {
            const C *tws = tw + (Ns - PPT) + (j & (Ns - 1));
#pragma unroll
            for (int r = 1; r < R; r++) x[r] = btw(x[r], TWG ? ldg(tws + (r - 1) * Ns) : tws[(r - 1) * Ns]);
        }
        if (LR == 3)
            bfly8<-1>(x);
        else if (LR == 2)
            bfly4<-1>(x[0], x[1], x[2], x[3]);
        else
            bfly2<-1>(x[0], x[1]);
#pragma unroll
        for (int r = 0; r < R; r++) v[b + NB * r] = last || (PPT == 4 && S == 2) ? bnorm(x[r]) : x[r];
    }
    if (!last) {
        if (!DB) seq_sync<WS>();
#pragma unroll
        for (int b = 0; b < NB; b++) {
            const int j = t + b * tps;
            const int d = ((j >> lNs) << (lNs + LR)) + (j & (Ns - 1));
#pragma unroll
            for (int r = 0; r < R; r++) buf[skew(d + r * Ns)] = v[b + NB * r];
        }
        seq_sync<WS>();
#pragma unroll
        for (int m = 0; m < PPT; m++) v[m] = buf[skew(t + tps * m)];
        if (DB) {
            C *o = buf;
            buf = buf2;
            buf2 = o;
        }
    }
}

template <int LOGN, int PPT, bool DB, bool WS, typename C>
__device__ __forceinline__ void fft_reg(C *v, C *&buf, C *&buf2, const C *__restrict__ tw, int t)
{
    constexpr int LP = PPT == 4 ? 2 : 3, NF = LOGN / LP, REM = LOGN % LP;
    if constexpr (PPT == 2) {
        static_assert(LOGN >= 6 && LOGN <= 8, "two stages of radix 8");
        C w1[2], w2[2];
        reg_twiddles2<LOGN, 3, 1>(w1, tw, t);
        if constexpr (REM > 0) reg_twiddles2<LOGN, REM, 2>(w2, tw, t);
        reg_stage2<LOGN, 3, 0, DB, WS>(v, buf, buf2, w1, t);
        reg_stage2<LOGN, 3, 1, DB, WS>(v, buf, buf2, w1, t);
        if constexpr (REM > 0) reg_stage2<LOGN, REM, 2, DB, WS>(v, buf, buf2, w2, t);
    } else {
        static_assert(NF >= 1 && NF <= 5, "one to five stages");
        reg_stage<LOGN, PPT, LP, 0, DB, WS>(v, buf, buf2, tw, t);
        if constexpr (NF > 1) reg_stage<LOGN, PPT, LP, 1, DB, WS>(v, buf, buf2, tw, t);
        if constexpr (NF > 2) reg_stage<LOGN, PPT, LP, 2, DB, WS>(v, buf, buf2, tw, t);
        if constexpr (NF > 3) reg_stage<LOGN, PPT, LP, 3, DB, WS>(v, buf, buf2, tw, t);
        if constexpr (NF > 4) reg_stage<LOGN, PPT, LP, 4, DB, WS>(v, buf, buf2, tw, t);
        if constexpr (REM > 0) reg_stage<LOGN, PPT, REM, NF, DB, WS>(v, buf, buf2, tw, t);
    }
}

__device__ __forceinline__ void prefetch_l2(const void *p, unsigned bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "r"(bytes) : "memory");
}

// slot of natural index e in a pair-layout row (the inverse of pair_kx)
__host__ __device__ __forceinline__ int pair_slot(int e, int N)
{
    return e < (N >> 1) ? 2 * e : (e == (N >> 1) ? 1 : 2 * (N - e) + 1);
}

// ---------------------------------------------------------------------------
template <typename T, int MODE, int LOGN>
__global__ void __launch_bounds__((RegCfg<T, LOGN, row_xf(MODE)>::row_threads), (RegCfg<T, LOGN, row_xf(MODE)>::row_minb))
row_pass_r(const fch_kparams kp)
{
    typedef typename CT<T>::t C;
    typedef RegCfg<T, LOGN, row_xf(MODE)> G;
    constexpr int N = G::N, PPT = G::ppt, TPS = G::tps;
    constexpr bool WS = TPS <= 32;
    constexpr bool INV = MODE != RM_R2C_LOAD && MODE != RM_NIMEX_DIRECT && MODE != RM_SAV_DIRECT;
    constexpr bool FWD = MODE != RM_C2R_STORE && MODE != RM_ENERGY;
    pdl_wait();
    if (G::early) pdl_trigger();
    if (pass_skipped(kp)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red_scratch[FCH_NRED * 32];
    if (kp.nfft && blockIdx.x == 0 && threadIdx.x == 0)
        atomicAdd(kp.nfft, (MODE == RM_R2C_LOAD || MODE == RM_C2R_STORE || MODE == RM_ENERGY) ? 2ull : 4ull);
    const C *tw = (const C *)(PPT == 4 ? kp.tw4 : kp.tw);
    const int rr = threadIdx.x / TPS, t = threadIdx.x % TPS, y = blockIdx.x * G::rpb + rr;
    C *buf = (C *)smem_raw + rr * G::SL, *buf2 = buf + (G::db ? G::rpb * G::SL : 0);
    C *Zrow = pair_Z<C>(kp, N) + (long)y * N;
    const bool f64io = kp.flags & FCH_FL_F64IO;
    const fch_consts<T> &K = consts<T>(kp);
    const long row0 = (long)y * N + t;

    C v[PPT];
    if (MODE == RM_NIMEX_DIRECT || MODE == RM_SAV_DIRECT) {
        // (u*, Lap u*) pointwise from the stored real-space slots (eq. Richardson)
        const fch_ctrl *cs = kp.ctrl;
        const C *Rn = (const C *)kp.Rs[cs->iu_n] + row0;
        const C *Rm = (const C *)kp.Rs[cs->iu_m] + row0;
        const T g = load_coef<T>(cs).gam;
        const bool plain = (kp.flags & FCH_FL_GAMMA0) || g == (T)0;
#pragma unroll
        for (int m = 0; m < PPT; m++) v[m] = ldg(Rn + TPS * m);
        if (!plain) {
#pragma unroll
            for (int m = 0; m < PPT; m++) v[m] = badd(v[m], lscale(bsub(v[m], ldg(Rm + TPS * m)), g));
        }
    } else if (MODE == RM_R2C_LOAD) {
        const void *in0 = pair_in(kp.in0, kp), *in1 = pair_in(kp.in1, kp);
        if (f64io) {
#pragma unroll
            for (int m = 0; m < PPT; m++) v[m].x = (T)((const double *)in0)[row0 + TPS * m];
#pragma unroll
            for (int m = 0; m < PPT; m++) v[m].y = in1 ? (T)((const double *)in1)[row0 + TPS * m] : (T)0;
        } else {
#pragma unroll
            for (int m = 0; m < PPT; m++) v[m].x = (T)((const float *)in0)[row0 + TPS * m];
#pragma unroll
            for (int m = 0; m < PPT; m++) v[m].y = in1 ? (T)((const float *)in1)[row0 + TPS * m] : (T)0;
        }
    } else {
#pragma unroll
        for (int m = 0; m < PPT; m++) v[m] = Zrow[pair_slot(t + TPS * m, N)];
    }

    T red[FCH_NRED] = {0, 0, 0, 0};
    constexpr bool PT = MODE != RM_R2C_LOAD && MODE != RM_C2R_STORE;
    constexpr bool has_red = MODE == RM_SAV || MODE == RM_SAV_DIRECT || MODE == RM_ENERGY;
    // the pointwise stage on the natural slots (and its block sums)
    auto pointwise_stage = [&]() {
        if (PT && PPT <= 4) {
#pragma unroll
            for (int m = 0; m < PPT; m++) v[m] = pointwise_elem<T, MODE>(kp, K, v[m], red);
        } else if (PT) {
            // eight points: through this thread's own natural slots (read last, or not yet
            // used), a loop of two points at a time instead of eight copies of the code
            C *own = G::db ? buf2 : buf;
#pragma unroll
            for (int m = 0; m < PPT; m++) own[skew(t + TPS * m)] = v[m];
#pragma unroll 2
            for (int m = 0; m < PPT; m++) {
                C *s = own + skew(t + TPS * m);
                *s = pointwise_elem<T, MODE>(kp, K, *s, red);
            }
#pragma unroll
            for (int m = 0; m < PPT; m++) v[m] = own[skew(t + TPS * m)];
        }
        if (has_red) {
            block_partials<1>(red, kp.part, red_scratch);
            if constexpr (row_tail_op(MODE) >= 0) pass_tail<row_tail_op(MODE)>(kp);
        }
    };
    if (!INV) pointwise_stage();
#pragma unroll 1
    for (int dir = INV ? 0 : 1; dir < (FWD ? 2 : 1); dir++) {
        if (INV && dir == 0) {
#pragma unroll
            for (int m = 0; m < PPT; m++) v[m].y = -v[m].y;
        }
        fft_reg<LOGN, PPT, G::db, WS>(v, buf, buf2, tw, t);
        if (INV && dir == 0) {
#pragma unroll
            for (int m = 0; m < PPT; m++) v[m].y = -v[m].y;
            if (MODE == RM_F && (kp.flags & FCH_FL_STORE_REAL)) {
                // F row pass of an adaptive trial: keep (u, Lap u) of this state in real space
                const fch_ctrl *cs = kp.ctrl;
                const int slot = kp.src == FCH_SRC_UNEW ? cs->iu_new : (kp.src == 5 ? cs->iu_m : cs->iu_n);
                C *store = (C *)kp.Rs[slot] + row0;
#pragma unroll
                for (int m = 0; m < PPT; m++) store[TPS * m] = v[m];
            }
            pointwise_stage();
        }
    }
    if (MODE == RM_C2R_STORE) {
        void *out0 = pair_out(kp.out0, kp), *out1 = pair_out(kp.out1, kp);
#pragma unroll
        for (int m = 0; m < PPT; m++) {
            const long g = row0 + TPS * m;
            if (f64io) {
                if (out0) ((double *)out0)[g] = (double)v[m].x;
                if (out1) ((double *)out1)[g] = (double)v[m].y;
            } else {
                if (out0) ((float *)out0)[g] = (float)v[m].x;
                if (out1) ((float *)out1)[g] = (float)v[m].y;
            }
        }
    }
    if (!G::early) pdl_trigger();
    if (FWD) {
#pragma unroll
        for (int m = 0; m < PPT; m++) Zrow[pair_slot(t + TPS * m, N)] = v[m];
    }
}

// ---------------------------------------------------------------------------
template <typename T, int MODE, int LOGN>
__device__ __forceinline__ void col_body_r(const fch_kparams &kp)
{
    typedef typename CT<T>::t C;
    typedef ColTraits<MODE> TR;
    typedef RegCfg<T, LOGN, col_xf(MODE)> G;
    namespace cg = cooperative_groups;
    constexpr int N = G::N, PPT = G::ppt, TPS = G::tps, H = PPT / 2;
    constexpr bool CL = G::cl, WS = G::col_threads <= 32;
    pdl_wait();
    if (G::early) pdl_trigger();
    if (pass_skipped(kp)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red_scratch[FCH_NRED * 32];
    const C *tw = (const C *)(PPT == 4 ? kp.tw4 : kp.tw);
    const fch_consts<T> &K = consts<T>(kp);
    const bool inv = TR::INV_ALWAYS || (TR::INV_OPT && (kp.flags & (FCH_FL_PACK_F | FCH_FL_PACK_USTAR)));
    const bool has_red = MODE == CM_SAV_PQ || MODE == CM_PSD_ITER ||
                         (MODE == CM_F_FINISH && (kp.flags & FCH_FL_AM3));
    // this thread's column: slot cc of the block's columns (slot c of pair p), point t + TPS m
    const int cc = CL ? 0 : (int)threadIdx.x % G::ncol, t = CL ? (int)threadIdx.x : (int)threadIdx.x / G::ncol;
    const int c = CL ? (int)(blockIdx.x & 1) : cc & 1;
    const int p = CL ? (int)(blockIdx.x >> 1) : (int)blockIdx.x * G::P + (cc >> 1);
    const bool has0 = CL ? p == 0 : blockIdx.x == 0; // the block holds pair 0
    C *buf = (C *)smem_raw + cc * G::SC, *buf2 = buf + (G::db ? G::ncol * G::SC : 0);
    // the partner column's buffer, as an offset from this column's, or its address in the
    // other block of the cluster
    C *Zc = pair_Z<C>(kp, N) + 2 * p + c;

    fch_coef<T> co;
    ColBufs<C> bf;
    load_colbufs<T>(kp, co, bf);

    if (G::prefetch && threadIdx.x == 0 && p > 0) {
        // the rows of spectra the spectral stage will read, on their way while the columns
        // transform (2048^2: 14.36 -> 14.19 ms, 1024^2 6.08 -> 6.02 ms with the unrolled items)
        constexpr bool un = MODE == CM_IMEX_SOLVE || MODE == CM_F_FINISH || MODE == CM_SAV_PQ || MODE == CM_PSD_ITER;
        constexpr bool um = MODE == CM_IMEX_SOLVE || MODE == CM_SAV_PQ || MODE == CM_PSD_ITER;
        constexpr int half = CL ? N / 2 : N;
        const long r = (long)p * N + (CL && c ? half : 0);
        if (un) prefetch_l2(bf.Un + r, half * sizeof(C));
        if (um) prefetch_l2(bf.Um + r, half * sizeof(C));
        if (MODE == CM_F_FINISH && has_red) {
            prefetch_l2(bf.src + r, half * sizeof(C));
            prefetch_l2(bf.Fn + r, half * sizeof(C));
            prefetch_l2(bf.Fm + r, half * sizeof(C));
        }
        if (MODE == CM_SAV_COMBINE) {
            prefetch_l2((const C *)kp.Pb + r, half * sizeof(C));
            prefetch_l2((const C *)kp.Qb + r, half * sizeof(C));
        }
    }
    C v[PPT];
    if (TR::FWD) {
        const unsigned m1 = c ? 0x80000000u : 0u; // column N - kx enters conjugated
#pragma unroll
        for (int m = 0; m < PPT; m++) v[m] = Zc[(long)(t + TPS * m) * N];
#pragma unroll
        for (int m = 0; m < PPT; m++) v[m].y = flip(v[m].y, m1);
    }

    T red[FCH_NRED] = {0, 0, 0, 0};
    auto pair_sync = [&]() { // the partner's slots are written (both threads of an item)
        if (CL)
            cg::this_cluster().sync();
        else if (has0)
            __syncthreads(); // pair 0 reads its own column's slots of other threads
        else
            __syncwarp();
    };
    auto spectral = [&]() {
        // the natural slots of the buffer read last (own slots: no other thread reads them
        // before the sync below); DB swapped the two after the last exchange
        C *own = G::db ? buf2 : buf;
        C *oth = CL ? cg::this_cluster().map_shared_rank(own, c ^ 1) : own + (c ? -G::SC : G::SC);
        if (TR::FWD) {
#pragma unroll
            for (int m = 0; m < PPT; m++) own[skew(t + TPS * m)] = v[m];
        }
        pair_sync();
        if (p > 0) {
            // column slot 0 takes the items m < H, slot 1 the others
            constexpr int UNR = G::items;
#pragma unroll UNR
            for (int i = 0; i < H; i++) {
                const int ky = t + TPS * (i + (c ? H : 0)), s = skew(ky);
                C A = mk<C>(0, 0), B = mk<C>(0, 0);
                if (TR::FWD) {
                    const C zo = own[s], zt = oth[s];
                    const C z0 = c ? zt : zo, w1 = c ? zo : zt; // Z(kx, ky), conj Z(N - kx, -ky)
                    A = cscale_p2(badd(z0, w1), (T)0.5);
                    const C dm = bsub(z0, w1);
                    B = mk<C>(mul_p2(dm.y, (T)0.5), mul_p2(dm.x, (T)-0.5));
                }
                C Co = mk<C>(0, 0), Do = mk<C>(0, 0);
                spec_elem<T, MODE>(kp, K, co, bf, p, ky, A, B, Co, Do, red);
                if (inv) {
                    // the inverse transforms run as conj, forward, conj; column N - kx in
                    // its conjugate: conj(C + i D) for slot 0, C* + i D* for slot 1
                    const C o0 = mk<C>(rsub(Co.x, Do.y), -radd(Co.y, Do.x));
                    const C o1 = mk<C>(radd(Co.x, Do.y), rsub(Do.x, Co.y));
                    own[s] = c ? o1 : o0;
                    oth[s] = c ? o0 : o1;
                }
            }
        } else {
            // columns 0 and N/2: item ky of a column pairs its rows ky and -ky; the thread of
            // index k takes item k of column 0, -k of column N/2 (held conjugated)
            C o[PPT];
#pragma unroll
            for (int m = 0; m < PPT; m++) o[m] = mk<C>(0, 0);
#pragma unroll
            for (int m = 0; m < PPT; m++) {
                const int k = t + TPS * m, mk_ = (N - k) & (N - 1);
                C A = mk<C>(0, 0), B = mk<C>(0, 0);
                if (TR::FWD) {
                    const C zk = own[skew(k)], zm = own[skew(mk_)];
                    // Z of the item's row and the conjugate of Z of the opposite row
                    const C za = c ? cconj(zk) : zk, zb = c ? zm : cconj(zm);
                    A = cscale_p2(badd(za, zb), (T)0.5);
                    const C dm = bsub(za, zb);
                    B = mk<C>(mul_p2(dm.y, (T)0.5), mul_p2(dm.x, (T)-0.5));
                }
                C Co = mk<C>(0, 0), Do = mk<C>(0, 0);
                spec_elem<T, MODE>(kp, K, co, bf, c ? N / 2 : 0, c ? mk_ : k, A, B, Co, Do, red);
                // column 0: conj(C + i D); column N/2, whose index k holds C + i D of item -k
                o[m] = mk<C>(rsub(Co.x, Do.y), radd(Co.y, Do.x));
                if (c == 0) o[m].y = -o[m].y;
            }
            if (inv) {
#pragma unroll
                for (int m = 0; m < PPT; m++) v[m] = o[m];
            }
        }
        if (has_red) {
            block_partials<2>(red, kp.part, red_scratch);
            if constexpr (col_tail_op(MODE) >= 0) pass_tail<col_tail_op(MODE)>(kp);
        }
        // results of the partner's items (and no block of a cluster leaves before its
        // partner has read it)
        if (CL || inv) pair_sync();
        if (inv && p > 0) {
#pragma unroll
            for (int m = 0; m < PPT; m++) v[m] = own[skew(t + TPS * m)];
        }
    };
    if (!TR::FWD) spectral();
#pragma unroll 1
    for (int dir = TR::FWD ? 0 : 1; dir < 2; dir++) {
        fft_reg<LOGN, PPT, G::db, WS>(v, buf, buf2, tw, t);
        if (TR::FWD && dir == 0) {
            spectral();
            if (!inv) return;
        }
    }
    if (!G::early) pdl_trigger();
    const unsigned m0 = c ? 0u : 0x80000000u;
#pragma unroll
    for (int m = 0; m < PPT; m++) {
        v[m].y = flip(v[m].y, m0);
        Zc[(long)(t + TPS * m) * N] = v[m];
    }
}

template <typename T, int MODE, int LOGN>
__global__ void __launch_bounds__((RegCfg<T, LOGN, col_xf(MODE)>::col_threads), (RegCfg<T, LOGN, col_xf(MODE)>::col_minb))
col_pass_r(const fch_kparams kp)
{
    col_body_r<T, MODE, LOGN>(kp);
}

// the same as clusters of two blocks, one column of a pair each
template <typename T, int MODE, int LOGN>
__global__ void __cluster_dims__(2, 1, 1)
    __launch_bounds__((RegCfg<T, LOGN, col_xf(MODE)>::col_threads), (RegCfg<T, LOGN, col_xf(MODE)>::col_minb))
col_pass_rcl(const fch_kparams kp)
{
    col_body_r<T, MODE, LOGN>(kp);
}

} // namespace fch
