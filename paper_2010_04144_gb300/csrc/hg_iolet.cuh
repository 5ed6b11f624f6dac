// hg_iolet.cuh -- what the per-step iolet update (hg_kernels.cu) and the resident multi-step
// kernel (hg_steps.cu) share: the FP64 terms, their order of summation and the boundary
// values that follow.  Explicit rounding intrinsics, so both produce the same bits.
#pragma once

#include "hg_internal.h"

namespace hg {
namespace {

// u.n and drho of one adjacent site's moments (drho, u).
__device__ __forceinline__ void iolet_terms(const IoDev &I, float4 m, double &su, double &sr) {
    su = __fma_rn((double)m.w, I.nz, __fma_rn((double)m.y, I.nx, __dmul_rn((double)m.z, I.ny)));
    sr = (double)m.x;
}
// Sums over a warp's lanes by a fixed tree, result in lane 0.
__device__ __forceinline__ void warp_sum2(double &a, double &b) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a = __dadd_rn(a, __shfl_down_sync(0xffffffffu, a, o));
        b = __dadd_rn(b, __shfl_down_sync(0xffffffffu, b, o));
    }
}
__device__ __forceinline__ double iolet_mean(const IoDev &I, double sum) {
    return I.n_slots ? __ddiv_rn(sum, (double)I.n_slots) : 0.0;
}
__device__ __forceinline__ void iolet_store_means(const IoDev &I, double mean_u, double sum_r) {
    I.M[0] = mean_u;
    I.M[1] = iolet_mean(I, sum_r);
    I.M[2] = (double)I.n_slots;
}
// The uncoupled boundary value for the step after step e: value x pulse.  Phase in [0, 1)
// by an exact remainder first, so the FP64 cosine only ever sees an argument in [0, 2 pi).
__device__ __noinline__ float iolet_value(const IoDev &I, int64_t e) {
    double p = 1.0;
    if (I.pulse) {
        const double x = __dmul_rn(6.283185307179586, fmod((double)(e + 1), I.period) / I.period);
        p = I.pulse == 1 ? __dmul_rn(0.5, __dsub_rn(1.0, cos(x))) : sin(x);
    }
    return (float)__dmul_rn(I.value, p);
}

}  // namespace
}  // namespace hg
