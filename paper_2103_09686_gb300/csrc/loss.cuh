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

// One thread: E, E^2, E_bc, lambda, L, rel_err and the gradient scalars from
// sum (D - D_des)^2, sum D_des^2 and the sum of the squared box excess; in a reconstruction
// also the stopping test and the Adam step bookkeeping.
__device__ __forceinline__ void loss_scalars(const LossSeg& sg, DF e2s, DF t2s, DF x2s) {
    const LossParams lp = sg.lp;
    Scalars* sc = sg.sc;
    float* loss_out = sg.loss_out;
    float* history = sg.history;
    // the scalars in FP64 on this one thread (a few dozen FP64 operations once per
    // evaluation): the double-float sums keep about 48 bits, and the square roots and
    // quotients below keep them, so E, rel_err and L reach the output rounded once to FP32
    const double E2 = (double)e2s.hi + (double)e2s.lo;
    const double T2 = (double)t2s.hi + (double)t2s.lo;
    const double ex2 = (double)x2s.hi + (double)x2s.lo;
    const double N = (double)lp.N;
    const double lam0 = lp.bc_on ? (double)lp.lambda0 : 0.0;
    const double E = sqrt(E2);
    const double Ebc = ex2 / (N * N);
    const double phi = lp.mode == 0 ? E : E2;
    const double lam = lam0 * phi;
    const double L = phi + lam * Ebc;
    const double rel = T2 > 0.0 ? E / sqrt(T2) : (double)INFINITY;
    const float out[6] = {(float)E, (float)E2, (float)Ebc, (float)lam, (float)L, (float)rel};
    for (int i = 0; i < 6; ++i) sc->loss[i] = out[i];
    if (loss_out != nullptr)
        for (int i = 0; i < 6; ++i) loss_out[i] = out[i];
    // dL/dD = phi'(E) (1 + lam0 E_bc) dE/dD ;  dL/dM (penalty) = lam0 phi dE_bc/dM
    double gs;
    if (lp.mode == 0) gs = E > 0.0 ? (1.0 + lam0 * Ebc) / E : 0.0;
    else gs = 2.0 * (1.0 + lam0 * Ebc);
    sc->gscale = (float)gs;
    sc->pen_coef = (float)(2.0 * lam0 * phi / (N * N));
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
    // beta^t products stay FP64: they are multiplied once per step over many steps
    const double b1t = sc->b1t * (double)lp.beta1;
    const double b2t = sc->b2t * (double)lp.beta2;
    sc->b1t = b1t;
    sc->b2t = b2t;
    sc->lr_t = (float)((double)lp.lr * sqrt(1.0 - b2t) / (1.0 - b1t));
}

// Whole block: sums the instance's block sums in a fixed order and finishes the loss.
__device__ __forceinline__ void loss_finish(const LossSeg& sg, DF* sh) {
    DF r2{0.f, 0.f}, t2{0.f, 0.f}, x2{0.f, 0.f};
    for (int i = threadIdx.x; i < sg.nsum; i += blockDim.x) {
        const float4 v = __ldcg(sg.sums + i);
        r2 = df_add(r2, DF{v.x, v.y});
        t2 = df_add(t2, DF{v.z, v.w});
    }
    for (int i = threadIdx.x; i < sg.nexc; i += blockDim.x) {
        const float4 v = __ldcg(sg.excess + i);
        x2 = df_add(x2, DF{v.x, v.y});
    }
    const DF e2s = block_sum_df(r2, sh);
    const DF t2s = block_sum_df(t2, sh);
    const DF x2s = block_sum_df(x2, sh);
    if (threadIdx.x == 0) loss_scalars(sg, e2s, t2s, x2s);
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
