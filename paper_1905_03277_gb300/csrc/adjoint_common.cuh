// Device functions shared by the adjoint's translation units (merge_bwd.cu,
// merge_bwd_region.cu).
#pragma once

#include <float.h>

#include "hmfsr_internal.cuh"

namespace hmfsr {
namespace {

// s + e plus o + oe, e and oe the rounding errors carried so far: s takes the rounded sum, e the
// errors and that rounding's exact error (two-sum)
__device__ __forceinline__ void two_sum(float &s, float &e, float o, float oe) {
    const float t = s + o, bp = t - s;
    e = (e + oe) + ((s - (t - bp)) + (o - bp));
    s = t;
}

// the error to go with a sum: none where the sum left the range (infinity less itself is no number)
__device__ __forceinline__ float error_of(float s, float e) { return fabsf(s) <= FLT_MAX ? e : 0.f; }

// Block sums in a fixed order without FP64 arithmetic per element (FP64 is scarce on this
// GPU): each warp (or group of kLanes) adds its lanes' values by butterflies carrying the exact
// rounding error of every FP32 addition, lane 0 stores the warp's (sum, error) pair; the
// caller's thread 0 then adds the warps' pairs in FP64 in warp order.
template <int K, int kLanes = 32>
__device__ __forceinline__ void warp_sums_comp(float (&v)[K], float (&e)[K]) {
#pragma unroll
    for (int q = 0; q < K; ++q) e[q] = 0.f;
#pragma unroll
    for (int o = kLanes / 2; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < K; ++q)
            two_sum(v[q], e[q], __shfl_xor_sync(0xffffffffu, v[q], o), __shfl_xor_sync(0xffffffffu, e[q], o));
#pragma unroll
    for (int q = 0; q < K; ++q) e[q] = error_of(v[q], e[q]);
}

// The six kernel parameters' contribution of one texel.  With k_x = s_x^2 the kernel
// variances of Eq. 4 / S.1 (s_along, s_across their square roots), d k_x / d p_q = 2 s_x
// a_x[q], and the texel adds sum_q (d k_across / d p_q bo1 + d k_along / d p_q bo2) to
// pb[q], bo1 and bo2 being dL/dk_across and dL/dk_along times the bilinear weight:
//   a_along  = {(1-D) k_stretch A + D k_denoise, D k_detail, (kd - kh_al) dD/dD_th,
//               (kd - kh_al) dD/dD_tr, (1-D) k_detail A, 0},
//   a_across = {(1-D) / (k_shrink A) + D k_denoise, D k_detail, (kd - kh_ac) dD/dD_th,
//               (kd - kh_ac) dD/dD_tr, 0, -(1-D) k_detail / (k_shrink^2 A)}
// with kd = k_detail k_denoise, kh_al = k_detail k_stretch A, kh_ac = k_detail /
// (k_shrink A), D = clamp(1 - sqrt(l1_norm) / D_tr + D_th, 0, 1) and its derivatives 0
// where clamped.  Per-call constants in KConsts; 1/A on the SFU.
struct KConsts {
    float inv_dtr, inv_shrink, kd, kds, kdi, kdi2;
};
__host__ __device__ __forceinline__ KConsts kconsts_of(const MergeConsts &c) {
    KConsts k;
    k.inv_dtr = 1.f / c.d_tr;
    k.inv_shrink = 1.f / c.k_shrink;
    k.kd = c.k_detail * c.k_denoise;
    k.kds = c.k_detail * c.k_stretch;
    k.kdi = c.k_detail * k.inv_shrink;
    k.kdi2 = k.kdi * k.inv_shrink;
    return k;
}
__device__ __forceinline__ void kernel_grad_acc(const float4 sh, const MergeConsts &c, const KConsts &k, float bo1,
                                                float bo2, float (&pb)[6]) {
    const float A = sh.x, rl = sh.y, invA = fast_rcp(A);
    const float Draw = 1.f - rl * k.inv_dtr + c.d_th;
    const float D = fminf(fmaxf(Draw, 0.f), 1.f), omD = 1.f - D;
    const bool inside = Draw > 0.f && Draw < 1.f;
    const float kh_al = k.kds * A, kh_ac = k.kdi * invA;
    const float s_al = omD * kh_al + D * k.kd, s_ac = omD * kh_ac + D * k.kd;
    const float P = 2.f * s_ac * bo1, Qv = 2.f * s_al * bo2;  // dL/d(a_across), dL/d(a_along) weights
    pb[0] = fmaf(P, omD * k.inv_shrink * invA + D * c.k_denoise, fmaf(Qv, omD * c.k_stretch * A + D * c.k_denoise, pb[0]));
    pb[1] = fmaf(P + Qv, D * c.k_detail, pb[1]);
    if (inside) {
        const float sD = P * (k.kd - kh_ac) + Qv * (k.kd - kh_al);
        pb[2] += sD;
        pb[3] = fmaf(sD, rl * k.inv_dtr * k.inv_dtr, pb[3]);
    }
    pb[4] = fmaf(Qv, omD * c.k_detail * A, pb[4]);
    pb[5] = fmaf(-P, omD * k.kdi2 * invA, pb[5]);
}

}  // namespace
}  // namespace hmfsr
