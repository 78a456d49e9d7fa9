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

// Double-precision reciprocal and sixth root: one step of third order from a
// single-precision seed (relative error e < 2^-21: the step leaves e^3, below double
// rounding). The controller is a chain of dependent operations on a slow double pipe, and
// a third-order step is three of them where two Newton steps are four (the root: nine
// where two Newton steps and the powers are sixteen).
__device__ inline double rcp_nr(double a)
{
    const double r = (double)(1.0f / (float)a), e = fma(-a, r, 1.0);
    return fma(r, fma(e, e, e), r); // 1/a = r / (1 - e) = r (1 + e + e^2 + ...)
}

// x^(1/6) for x in [1e-30, 1e30]: z = x^(-1/6) from a seed, with d = 1 - x z^6 the root is
// z (1 - d)^(-1/6) = z (1 + d/6 + 7 d^2/72 + ...); then x z^5
__device__ inline double root6_nr(double x)
{
    const double z = (double)powf((float)x, -1.0f / 6.0f);
    const double z2 = z * z, z4 = z2 * z2;
    const double d = fma(-x, z4 * z2, 1.0);
    const double y = fma(z * d, fma(d, 7.0 / 72.0, 1.0 / 6.0), z);
    const double y2 = y * y;
    return (x * y) * (y2 * y2);
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
        if (!isfinite(v) || v <= 0) {
            c->status = FCH_ENONFINITE;
            c->done = 1;
            return false;
        }
        c->e1 = e1;
        c->inv_sqrt_e1 = 1.0 / sqrt(v);
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
        const double ratio = sqrt(S0) / sqrt(S1); // ||d|| / ||v_{s+1}||, h cancels
        c->psd_iter++;
        c->n_psd_iter++;
        c->psd_ratio = ratio;
        if (!isfinite(ratio)) {
            c->status = FCH_ENONFINITE;
            c->done = 1;
        } else if (S0 < c->itol * c->itol * S1) {
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
        // A_dp = rho_s k (sigma/e)^(1/3) = rho_s k (sigma^2 S1 / S0)^(1/6), e >= 1e-16
        c->n_attempts++;
        if (!isfinite(S0) || !isfinite(S1) || !(S1 > 0)) {
            c->status = FCH_ENONFINITE;
            c->done = 1;
            return false;
        }
        c->lte_num = S0;
        c->lte_den = S1;
        const double k1 = c->k1;
        const double x = fmin(c->sigma2 * S1 * rcp_nr(fmax(S0, 1e-32 * S1)), 1e30);
        double kn = c->rho_s * k1 * root6_nr(x);
        if (c->cap) kn = fmin(kn, 2.414213562373095 * k1); // (1 + sqrt 2) k
        kn = fmax(c->kmin, fmin(kn, c->kmax));
        if (S0 <= c->sigma2 * S1 || k1 <= c->kmin) {
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

// The set-up of a trial of size arg0 (fixed step) or, where arg0 <= 0, of the next adaptive
// trial: by one warp. Lane 0 has run whatever came before; the lanes compute the same
// coefficients, and ten of them look the PSD search step up at once.
__device__ __forceinline__ void ctrl_init_trial(fch_ctrl *c, double arg0, int lane)
{
    double k1;
    if (arg0 > 0) {
        k1 = arg0; // fixed step
    } else {
        const double rem = c->t_final - c->t;
        if (rem <= 1e-12 * fmax(1.0, fabs(c->t_final))) {
            __syncwarp();
            c->done = 1;
            return;
        }
        k1 = fmin(c->ktrial, rem); // the run ends exactly at t_final
    }
    const double kn = c->kn;
    double a, b, cc, g, w1 = c->w1, w2 = c->w2, w3 = c->w3;
    if (kn <= 0) { // backward-Euler start: k_{n-1} -> infinity in eq. (BDF2Coef)
        a = rcp_nr(k1);
        b = -a;
        cc = 0.0;
        g = 0.0;
    } else {
        // eq. (BDF2Coef) and the eq. (Predictor) weights from three independent
        // reciprocals (1/(1+gam) = k_n/(k_{n+1}+k_n)), so their latencies overlap
        const double r1 = rcp_nr(k1), rn = rcp_nr(kn), rs = rcp_nr(k1 + kn);
        a = r1 + rs;
        b = -r1 - rn;
        cc = rn - rs;
        g = k1 * rn;
        const double k6 = k1 * (1.0 / 6.0), ig = kn * rs; // 1/(1+g)
        w1 = k6 * (3.0 + 2.0 * g) * ig;
        w2 = k6 * (3.0 + g);
        w3 = -k6 * g * g * ig;
    }
    // PSD search step: Table SearchSize row, linear in k, clamped (slopes precomputed)
    const unsigned above = __ballot_sync(0xffffffffu, lane < 10 && k1 > c->lam_k[lane < 10 ? lane : 0]);
    const int j = c->lam_k[0] < 0 ? -1 : __popc(above) - 1; // last knot below k1
    double lam;
    if (j < 0)
        lam = c->lam_tab[0];
    else if (k1 >= c->lam_k[9])
        lam = c->lam_tab[9];
    else
        lam = c->lam_tab[j] + (k1 - c->lam_k[j]) * c->lam_slope[j];
    __syncwarp(); // every lane has read the old values
    if (lane == 0) {
        c->k1 = k1;
        c->a = a;
        c->b = b;
        c->c = cc;
        c->gam = g;
        c->w1 = w1;
        c->w2 = w2;
        c->w3 = w3;
        c->lam = lam;
        c->psd_conv = 0;
        c->psd_iter = 0;
    }
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

// The whole control step by one block (any multiple of 32 threads up to 1024): the control
// block is staged through shared memory with coalesced copies, the first na partials of
// the slots the operation reads are summed in a fixed order, warp 0 runs the operation, and
// the block writes the control block back. What it costs is double-precision instructions
// (one warp instruction holds the pipe 16 cycles whatever its lanes do) and their chains:
// both slots are reduced in the two halves of a warp at once, and the warp sums by a second
// shuffle tree.
template <int OP> __device__ __forceinline__ void ctrl_block(const fch_kparams &kp, int na, double arg0)
{
    constexpr int slots = ctrl_slots<OP>();
    __shared__ double sh[2][32];
    __shared__ fch_ctrl cs;
    const int nw = (int)(sizeof(fch_ctrl) / 8);
    const int nthr = blockDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < nw; i += nthr) ((long long *)&cs)[i] = ((const long long *)kp.ctrl)[i];
    // the partial sums load while the control block arrives (discarded if it says done)
    double s0 = 0, s1 = 0;
    if (slots > 0) {
        for (int i = threadIdx.x; i < na; i += 4 * nthr) {
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
            const int w = nthr >> 5, l = lane & 15, h = lane >> 4;
            double v = l < w ? sh[h][l] : 0.0;
            if (w > 16) v += l + 16 < w ? sh[h][l + 16] : 0.0;
            for (int o = 8; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o, 16);
            S0 = __shfl_sync(0xffffffffu, v, 0);
            S1 = __shfl_sync(0xffffffffu, v, 16);
        }
        // the combined operations: the decision (adaptive) or the acceptance of a fixed
        // step, then the set-up of the next trial (adaptive: -1; fixed: arg0 = dt)
        constexpr int FIRST = OP == OP_DECIDE_INIT ? OP_DECIDE : OP == OP_ACCEPT_INIT ? OP_ACCEPT : OP;
        bool go = true;
        if (FIRST != OP_INIT_TRIAL) {
            if (lane == 0) go = ctrl_op<FIRST>(&cs, kp, S0, S1, OP == OP_ACCEPT_INIT ? 0.0 : arg0);
            go = __shfl_sync(0xffffffffu, go, 0);
        }
        __syncwarp();
        if ((OP == OP_INIT_TRIAL || OP == OP_DECIDE_INIT || OP == OP_ACCEPT_INIT) && go)
            ctrl_init_trial(&cs, OP == OP_DECIDE_INIT ? -1.0 : arg0, lane);
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
