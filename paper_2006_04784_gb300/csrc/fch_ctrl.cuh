// fch_ctrl.cuh -- the device-side control logic of the adaptive steppers:
// FP64 reductions of per-block partial sums, the step-size controller of
// Sec. 3.2, the SAV scalar update and the PSD stopping test. Run either by the
// single-block control kernel or by the last block of the pass that produced
// the partial sums.
#pragma once
#include <math.h>
#include <stddef.h>
#include "fch_internal.h"
#include "../../include/fch.h"

// Programmatic dependent launch: the passes and the control kernel are launched
// with programmatic stream serialization, so a launch may begin while its
// predecessor in the stream drains. Every kernel first waits for the predecessor to
// complete (its writes visible), before it reads anything, then allows its own
// successor to begin launching; the successor's blocks wait in turn. Launched
// without the attribute, both instructions return at once.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_begin()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// What the control steps cost is double-precision instructions: on this GPU one of them
// holds an SM's sub-partition for 64 cycles, whatever its lanes do and whether or not it
// depends on the one before (conversions too; fmin 155, a division 365, a square root 610:
// measured). So few of them, spread over warps of different sub-partitions where they are
// independent, and comparisons on the bits: doubles that are not negative are ordered as
// their bit patterns are, and so is any number against one that is not. Against chains of
// one warp with double comparisons and two square roots a check: 24 PSD trials of 256^2 in
// double-float 2618 -> 2534 us, 32 IMEX trials of 512^2 with the regularised well 1662 ->
// 1605 us.
__device__ __forceinline__ long long ord(double a) { return __double_as_longlong(a); }
__device__ __forceinline__ double pmin(double a, double b) { return ord(a) < ord(b) ? a : b; }
__device__ __forceinline__ double pmax(double a, double b) { return ord(a) > ord(b) ? a : b; }

// Double-precision reciprocal and x^(-1/6): one step of third order from a single-precision
// seed (relative error e < 2^-21: the step leaves e^3, below double rounding).
__device__ inline double rcp_nr(double a)
{
    const double r = (double)(1.0f / (float)a), e = fma(-a, r, 1.0);
    return fma(r, fma(e, e, e), r); // 1/a = r / (1 - e) = r (1 + e + e^2 + ...)
}

// x in [1e-30, 1e36]: with a seed z and d = 1 - x z^6 the root is z (1 - d)^(-1/6) =
// z (1 + d/6 + 7 d^2/72 + ...)
__device__ inline double rroot6_nr(double x)
{
    const double z = (double)powf((float)x, -1.0f / 6.0f);
    const double z2 = z * z, z4 = z2 * z2;
    const double d = fma(-x, z4 * z2, 1.0);
    return fma(z * d, fma(d, 7.0 / 72.0, 1.0 / 6.0), z);
}

// one control operation; returns false when the run stopped (done or failure). The
// operation is a template argument: a kernel holds the code (and the registers) of the
// operations it can run only.
template <int OP>
__device__ __forceinline__ bool ctrl_op(fch_ctrl *c, const fch_kparams &kp, double S0, double S1, double arg0)
{
    if constexpr (OP == OP_SAV_E1) {
        const double e1 = kp.h2 * S0;
        const double v = e1 + kp.D0;
        if (!isfinite(v) || ord(v) <= 0) {
            c->status = FCH_ENONFINITE;
            c->done = 1;
            return false;
        }
        c->e1 = e1;
        c->inv_sqrt_e1 = rsqrt(v);
        if (arg0 == 1.0) c->r_n = sqrt(v);
        if (arg0 == 2.0) c->r_m = sqrt(v);
    } else if constexpr (OP == OP_SAV_R) {
        // eq. (4.8) with u^{n+1} = p + r q:
        // r (a - a (X, q)/2) = -b r^n - c r^{n-1} + (X, a p + b u^n + c u^{n-1})/2
        const double sc = kp.h2 * kp.inv_n2; // Parseval on the unnormalised half spectra
        const double xr = sc * S0, xq = sc * S1;
        const double r = (-c->b * c->r_n - c->c * c->r_m + 0.5 * xr) / (c->a * (1.0 - 0.5 * xq));
        if (!isfinite(r)) {
            c->status = FCH_ENONFINITE;
            c->done = 1;
            return false;
        }
        c->r_new = r;
    } else if constexpr (OP == OP_PSD_CHECK) {
        // ||d|| / ||v_{s+1}|| < i_tol on the squares (h cancels)
        c->psd_iter++;
        c->n_psd_iter++;
        if (!isfinite(S0) || !isfinite(S1) || !(ord(S1) > 0)) {
            c->status = FCH_ENONFINITE;
            c->done = 1;
        } else if (ord(S0) < ord(c->itol * c->itol * S1)) {
            c->psd_conv = 1;
            c->last_psd_iter = c->psd_iter;
        } else if (c->psd_iter >= c->psd_max_iter) {
            c->status = FCH_ENOCONV;
            c->done = 1;
            c->last_psd_iter = c->psd_iter;
        }
    } else if constexpr (OP == OP_DECIDE) {
        // Steps 3-4 of the adaptive algorithm, Sec. 3.2, with e^2 = S0/S1:
        // accept iff S0 <= sigma^2 S1 (or k <= k_min);
        // A_dp = rho_s k (sigma/e)^(1/3) = rho_s k (S0 / (sigma^2 S1))^(-1/6), e >= 1e-16
        c->n_attempts++;
        if (!isfinite(S0) || !isfinite(S1) || !(ord(S1) > 0)) {
            c->status = FCH_ENONFINITE;
            c->done = 1;
            return false;
        }
        c->lte_num = S0;
        c->lte_den = S1;
        const double k1 = c->k1, m = c->sigma2 * S1;
        const double x = pmin(pmax(pmax(S0, 1e-32 * S1) * rcp_nr(pmax(m, 1e-36)), 1e-30), 1e36);
        double kn = c->rho_s * k1 * rroot6_nr(x);
        if (c->cap) kn = pmin(kn, 2.414213562373095 * k1); // (1 + sqrt 2) k
        kn = pmax(c->kmin, pmin(kn, c->kmax));
        if (ord(S0) <= ord(m) || ord(k1) <= ord(c->kmin)) {
            const int un = c->iu_n, um = c->iu_m, fn = c->if_n, fm = c->if_m;
            c->iu_m = un;
            c->iu_n = c->iu_new;
            c->iu_new = um;
            c->if_m = fn;
            c->if_n = c->if_new;
            c->if_new = fm;
            c->r_m = c->r_n;
            c->r_n = c->r_new;
            c->kn = k1;
            c->t += k1;
            c->n_steps++;
            c->accepted_last = 1;
        } else {
            c->n_rejects++;
            c->accepted_last = 0;
        }
        c->ktrial = kn;
    } else if constexpr (OP == OP_ACCEPT) {
        const int un = c->iu_n, um = c->iu_m;
        c->iu_m = un;
        c->iu_n = c->iu_new;
        c->iu_new = um;
        if (arg0 == 1.0) { // also rotate the F history (adaptive start)
            const int fn = c->if_n, fm = c->if_m;
            c->if_m = fn;
            c->if_n = c->if_new;
            c->if_new = fm;
        }
        c->r_m = c->r_n;
        c->r_n = c->r_new;
        c->kn = c->k1;
        c->ktrial = c->k1;
        c->t += c->k1;
        c->n_steps++;
        c->n_attempts++;
    } else if constexpr (OP == OP_ENERGY) {
        c->energy = kp.h2 * S0;
    }
    return !c->done;
}

// The size of the next trial: arg0 (fixed step), or the controller's proposal clipped so
// that the run ends exactly at t_final; 0 where it has ended (done is set).
__device__ __forceinline__ double ctrl_next_size(fch_ctrl *c, double arg0)
{
    if (arg0 > 0) return arg0;
    const double rem = c->t_final - c->t;
    if (ord(rem) <= ord(1e-12 * pmax(1.0, fabs(c->t_final)))) {
        c->done = 1;
        return 0.0;
    }
    return pmin(c->ktrial, rem);
}

// The set-up of a trial of size k1, by the first four warps of a block (each on a
// sub-partition of its own; every thread of the block calls it): eq. (BDF2Coef), the eq.
// (Predictor) weights and the PSD search step.
__device__ __forceinline__ void ctrl_init_trial(fch_ctrl *c, double k1, int warp, int lane)
{
    __shared__ double iv[5]; // 1/k1, 1/(k1 + kn), 1/kn, gam, k1/6
    const double kn = c->kn;
    const bool start = ord(kn) <= 0; // backward-Euler start: k_{n-1} -> infinity in eq. (BDF2Coef)
    double v = 0.0;
    if (warp == 0) {
        v = rcp_nr(k1);
        if (lane == 0) iv[0] = v;
    } else if (warp == 1 && !start) {
        v = rcp_nr(k1 + kn); // 1/(1+gam) = k_n/(k_{n+1}+k_n)
        if (lane == 0) iv[1] = v;
    } else if (warp == 2 && !start) {
        v = rcp_nr(kn);
        const double g = k1 * v;
        if (lane == 0) {
            iv[2] = v;
            iv[3] = g;
        }
    } else if (warp == 3) {
        if (lane == 0) iv[4] = k1 * (1.0 / 6.0);
        // Table SearchSize row, linear in k, clamped (slopes precomputed); ten lanes look it up
        const unsigned above =
            __ballot_sync(0xffffffffu, lane < 10 && ord(k1) > ord(c->lam_k[lane < 10 ? lane : 0]));
        const int j = ord(c->lam_k[0]) < 0 ? -1 : __popc(above) - 1; // last knot below k1
        if (lane == 0)
            c->lam = j < 0                           ? c->lam_tab[0]
                     : ord(k1) >= ord(c->lam_k[9]) ? c->lam_tab[9]
                                                     : c->lam_tab[j] + (k1 - c->lam_k[j]) * c->lam_slope[j];
    }
    __syncthreads();
    if (lane == 0 && warp < 4) {
        const double r1 = iv[0], rs = iv[1], rn = iv[2], g = iv[3], k6 = iv[4];
        if (warp == 0) {
            c->k1 = k1;
            c->psd_conv = 0;
            c->psd_iter = 0;
            c->a = start ? r1 : r1 + rs;
            c->c = start ? 0.0 : rn - rs;
            if (!start) c->w2 = k6 * (3.0 + g);
        } else if (warp == 1) {
            c->gam = start ? 0.0 : g;
            c->b = start ? -r1 : -r1 - rn;
        } else if (!start) {
            const double ig = kn * rs; // 1/(1+g)
            if (warp == 2)
                c->w1 = k6 * (3.0 + 2.0 * g) * ig;
            else
                c->w3 = -k6 * g * g * ig;
        }
    }
    __syncthreads();
}

// Float, double and double-float mirrors of the per-trial coefficients read by
// the passes, lane i of the calling warp converting coefficient i: conversions run
// on the double pipe, where one warp instruction costs the same for eleven lanes as
// for one, so the eleven conversions cost one instruction sequence instead of eleven.
static_assert(offsetof(fch_ctrl, lam) == offsetof(fch_ctrl, a) + 7 * sizeof(double),
              "a, b, c, gam, w1, w2, w3, lam are consecutive doubles");
static_assert(sizeof(fch_coef<float>) == 11 * sizeof(float) && sizeof(fch_coef<double>) == 11 * sizeof(double) &&
                  sizeof(fch_coef<fch::df>) == 11 * sizeof(fch::df),
              "fch_coef is eleven coefficients in declaration order");
__device__ inline void sync_coef_lanes(fch_ctrl *c, int lane)
{
    if (lane < 11) {
        const double v = lane < 8 ? (&c->a)[lane] : lane == 8 ? c->k1 : lane == 9 ? c->r_new : c->inv_sqrt_e1;
        ((float *)&c->cof)[lane] = (float)v;
        ((double *)&c->cod)[lane] = v;
        ((fch::df *)&c->codf)[lane] = fch::df(v);
    }
}


// block sums an operation reads: slots 0 and 1, slot 0, or none
template <int OP> constexpr int ctrl_slots()
{
    return OP == OP_DECIDE_INIT || OP == OP_SAV_R || OP == OP_PSD_CHECK ? 2 : OP == OP_SAV_E1 || OP == OP_ENERGY ? 1 : 0;
}

// The whole control step by one block (any multiple of 32 threads up to 1024; the set-up of
// a trial, 128 or more): the control block is staged through shared memory with coalesced
// copies, the first na partials of the slots the operation reads are summed in a fixed
// order, warp 0 runs the operation, and the block writes the control block back. Both slots
// are reduced in the two halves of a warp at once, by the warps that hold partials.
template <int OP> __device__ __forceinline__ void ctrl_block(const fch_kparams &kp, int na, double arg0)
{
    constexpr int slots = ctrl_slots<OP>();
    constexpr bool init = OP == OP_INIT_TRIAL || OP == OP_DECIDE_INIT || OP == OP_ACCEPT_INIT;
    __shared__ double sh[2][32];
    __shared__ fch_ctrl cs;
    __shared__ double k1s;
    const int nw = (int)(sizeof(fch_ctrl) / 8);
    const int nthr = blockDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < nw; i += nthr) ((long long *)&cs)[i] = ((const long long *)kp.ctrl)[i];
    // the partial sums load while the control block arrives (discarded if it says done)
    const int wact = min((na + 31) >> 5, nthr >> 5); // warps with partials
    if (slots > 0 && warp < wact) {
        const int i0 = threadIdx.x;
        double s0 = i0 < na ? kp.part[i0] : 0.0, s1 = slots > 1 && i0 < na ? kp.part[FCH_MAXBLK + i0] : 0.0;
        for (int i = i0 + nthr; i < na; i += 4 * nthr) {
            double v0[4], v1[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const int j = i + k * nthr;
                v0[k] = j < na ? kp.part[j] : 0.0;
                v1[k] = slots > 1 && j < na ? kp.part[FCH_MAXBLK + j] : 0.0;
            }
#pragma unroll
            for (int k = 0; k < 4; k++) {
                if (i + k * nthr >= na) break;
                s0 += v0[k];
                if (slots > 1) s1 += v1[k];
            }
        }
        // lanes 0-15 go on with slot 0, lanes 16-31 with slot 1
        double v = lane < 16 ? s0 : s1;
        v += __shfl_xor_sync(0xffffffffu, lane < 16 ? s1 : s0, 16);
        for (int o = 8; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o, 16);
        if ((lane & 15) == 0) sh[lane >> 4][warp] = v;
    }
    __syncthreads();
    if (cs.done && !(kp.flags & FCH_FL_NOSKIP)) return;
    if (OP == OP_PSD_CHECK && cs.psd_conv) return;
    if (warp == 0) {
        double S0 = 0, S1 = 0;
        if (slots > 0) {
            const int l = lane & 15, h = lane >> 4;
            double v = l < wact ? sh[h][l] : 0.0;
            if (wact > 16) v += l + 16 < wact ? sh[h][l + 16] : 0.0;
            for (int o = 8; o > 0; o >>= 1)
                if (o < wact) v += __shfl_down_sync(0xffffffffu, v, o, 16);
            S0 = __shfl_sync(0xffffffffu, v, 0);
            S1 = __shfl_sync(0xffffffffu, v, 16);
        }
        // the combined operations: the decision (adaptive) or the acceptance of a fixed
        // step, then the set-up of the next trial (adaptive: -1; fixed: arg0 = dt)
        constexpr int FIRST = OP == OP_DECIDE_INIT ? OP_DECIDE : OP == OP_ACCEPT_INIT ? OP_ACCEPT : OP;
        if (lane == 0) {
            bool go = true;
            if (FIRST != OP_INIT_TRIAL) go = ctrl_op<FIRST>(&cs, kp, S0, S1, OP == OP_ACCEPT_INIT ? 0.0 : arg0);
            if (init) k1s = go ? ctrl_next_size(&cs, OP == OP_DECIDE_INIT ? -1.0 : arg0) : 0.0;
        }
    }
    if (init) {
        __syncthreads();
        const double k1 = k1s;
        if (ord(k1) > 0) ctrl_init_trial(&cs, k1, warp, lane);
    }
    if (warp == 0) {
        __syncwarp();
        sync_coef_lanes(&cs, lane);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nw; i += nthr) ((long long *)kp.ctrl)[i] = ((const long long *)&cs)[i];
}

// Called by every block of a pass after its partial sums are written (where the launch
// asks for it, kp.tail_op >= 0): the last block to arrive (atomic ticket after a fence)
// runs the control operation of the pass over the partials of all gridDim.x blocks, then
// resets the ticket.
template <int OP> __device__ __forceinline__ void pass_tail(const fch_kparams &kp)
{
    if (kp.tail_op < 0) return;
    __shared__ unsigned int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(kp.ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    ctrl_block<OP>(kp, gridDim.x, kp.tail_arg);
    if (threadIdx.x == 0) *kp.ticket = 0;
}
