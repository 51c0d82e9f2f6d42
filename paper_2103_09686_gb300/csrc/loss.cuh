// The loss of one evaluation (Sec. 3.1, Eq. L_func_dMCR) from its three sums, and the last-block
// scheme by which the kernels that write a descriptor finish it without another launch.
#pragma once
#include <math.h>

#include "common.cuh"

namespace dmcr {

// Kahan sum
__device__ __forceinline__ void kahan_add(float& sum, float& comp, float v) {
    const float y = v - comp;
    const float t = sum + y;
    comp = (t - sum) - y;
    sum = t;
}

// Box excess of Sec. 3.1: (M-1) H(M-1) - M H(-M), H(0) = 0.
__device__ __forceinline__ float box_excess(float M) {
    return M > 1.f ? M - 1.f : (M < 0.f ? -M : 0.f);
}

// Warp 0: E, E^2, E_bc, lambda, L, rel_err and the gradient scalars from
// sum (D - D_des)^2, sum D_des^2 and the sum of the squared box excess; in a reconstruction
// also the stopping test and the Adam step bookkeeping.
// In FP64: the double-float sums keep about 48 bits, and the square roots and quotients below
// keep them, so E, rel_err and L reach the output rounded once to FP32.  An FP64 root or quotient
// is a chain of several hundred cycles and every other block waits for this one, so a lane each
// takes the three roots, then the four quotients that depend on nothing else, at once.
__device__ __forceinline__ void loss_scalars(const LossSeg& sg, DF e2s, DF t2s, DF x2s) {
    const LossParams& lp = sg.lp;
    Scalars* sc = sg.sc;
    const int lane = threadIdx.x & 31;
    const double E2 = (double)e2s.hi + (double)e2s.lo;
    const double T2 = (double)t2s.hi + (double)t2s.lo;
    const double ex2 = (double)x2s.hi + (double)x2s.lo;
    const double N = (double)lp.N;
    const double lam0 = lp.bc_on ? (double)lp.lambda0 : 0.0;
    // beta^t products stay FP64: they are multiplied once per step over many steps
    const double b1t = sc->b1t * (double)lp.beta1;
    const double b2t = sc->b2t * (double)lp.beta2;
    const double root = sqrt(lane == 0 ? E2 : (lane == 1 ? T2 : 1.0 - b2t));
    const double E = __shfl_sync(0xffffffffu, root, 0);
    const double rootT = __shfl_sync(0xffffffffu, root, 1), rootB = __shfl_sync(0xffffffffu, root, 2);
    const double phi = lp.mode == 0 ? E : E2;
    const double lam = lam0 * phi;
    // E / |D_des|, E_bc, the penalty's gradient factor, Adam's step
    const double num = lane == 0 ? E : (lane == 1 ? ex2 : (lane == 2 ? 2.0 * lam0 * phi : (double)lp.lr * rootB));
    const double den = lane == 0 ? rootT : (lane <= 2 ? N * N : 1.0 - b1t);
    const double quot = num / den;
    const double Ebc = __shfl_sync(0xffffffffu, quot, 1);
    const float pen_coef = (float)__shfl_sync(0xffffffffu, quot, 2);
    const float lr_t = (float)__shfl_sync(0xffffffffu, quot, 3);
    if (lane != 0) return;
    const double L = phi + lam * Ebc;
    const double rel = T2 > 0.0 ? quot : (double)INFINITY;
    // dL/dD = phi'(E) (1 + lam0 E_bc) dE/dD ;  dL/dM (penalty) = lam0 phi dE_bc/dM
    double gs;
    if (lp.mode == 0) gs = E > 0.0 ? (1.0 + lam0 * Ebc) / E : 0.0;
    else gs = 2.0 * (1.0 + lam0 * Ebc);
    sc->gscale = (float)gs;
    sc->pen_coef = pen_coef;
    float* loss_out = sg.loss_out;
    float* history = sg.history;
    const float out[6] = {(float)E, (float)E2, (float)Ebc, (float)lam, (float)L, (float)rel};
    for (int i = 0; i < 6; ++i) sc->loss[i] = out[i];
    if (loss_out != nullptr)
        for (int i = 0; i < 6; ++i) loss_out[i] = out[i];
    if (!lp.recon) return;
    const int it = sc->iter;
    if (history != nullptr && it < lp.max_iters) {
        history[3 * it + 0] = out[0];
        history[3 * it + 1] = out[4];
        history[3 * it + 2] = out[5];
    }
    sc->iter = it + 1;
    if (!isfinite(out[4])) { sc->done = 2; return; }
    if (lp.tol_rel > 0.f && (it % lp.check_every) == 0 && out[5] < lp.tol_rel) { sc->done = 1; return; }
    if (it + 1 > lp.max_iters) { sc->done = 3; return; }
    sc->adam_step = sc->adam_step + 1;
    sc->b1t = b1t;
    sc->b2t = b2t;
    sc->lr_t = lr_t;
}

// Whole block: sums the instance's block sums in a fixed order and finishes the loss.  `sh`: three
// entries for every warp.
__device__ __forceinline__ void loss_finish(const LossSeg& sg, DF* sh) {
    DF v[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    for (int i = threadIdx.x; i < sg.nsum; i += blockDim.x) {
        const float4 s = __ldcg(sg.sums + i);
        v[0] = df_add(v[0], DF{s.x, s.y});
        v[1] = df_add(v[1], DF{s.z, s.w});
    }
    for (int i = threadIdx.x; i < sg.nexc; i += blockDim.x) {
        const float4 s = __ldcg(sg.excess + i);
        v[2] = df_add(v[2], DF{s.x, s.y});
    }
    block_sums_df(v, sh);
    if (threadIdx.x < 32) loss_scalars(sg, v[0], v[1], v[2]);
}

// Called by every block (all threads) of the launch that leaves an instance's `count` block
// sums, after its own are written by thread 0: the block that arrives last finishes the loss.
// Its order of summation does not depend on which block that is.
__device__ __forceinline__ void loss_arrive(const LossSeg& sg, int count, DF* sh) {
    __shared__ int last;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&sg.sc->ticket, 1u) == (unsigned)count - 1u;
        if (last) {
            sg.sc->ticket = 0;
            __threadfence();
        }
    }
    __syncthreads();
    if (last) loss_finish(sg, sh);
}

}  // namespace dmcr
