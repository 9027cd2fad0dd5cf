// The noise model's uses beyond the closed form.  Noise-dependent tuning (supplement,
// "Noise-dependent Tuning" and "Tuning Procedure and Parameters"): the base frame's mean
// brightness and the noise model give an SNR, and the kernel parameters and the tile size
// follow from it.  Monte-Carlo noise statistics (Sec. 5.2.2): the robustness's modelled
// sigma_md^2 and d_md^2 per brightness level, simulated with rounding and clipping.
//
// The mean comes from an exact integer sum of the frame's samples on the GPU
// (hmfsr_frame_sum); the mapping from SNR to parameters is host arithmetic
// (hmfsr_snr_tuning).
#include <cooperative_groups.h>
#include <math.h>

#include "hmfsr_internal.cuh"

namespace hmfsr {
namespace {

constexpr int kSumThreads = 256, kSumPerThread = 8;

// Sum of every sample of one frame into *sum (zeroed by the caller's stream first).
// Thread t of block (bx, by) reads 8 consecutive samples of the rows by, by + gridDim.y,
// ..., four rows at a time so that four loads are in flight; the partial sums are exact in
// 64 bits and the atomic adds of exact integers commute, so the result does not depend on
// the order.
__device__ __forceinline__ unsigned int sum8(uint4 v) {
    return (v.x & 0xffffu) + (v.x >> 16) + (v.y & 0xffffu) + (v.y >> 16) + (v.z & 0xffffu) + (v.z >> 16) +
           (v.w & 0xffffu) + (v.w >> 16);
}

__global__ void __launch_bounds__(kSumThreads) k_frame_sum(const uint16_t *__restrict__ fr, int h, int w, int pitch,
                                                           unsigned long long *__restrict__ sum) {
    const int x0 = (blockIdx.x * kSumThreads + threadIdx.x) * kSumPerThread;
    const int gy = gridDim.y;
    unsigned long long acc = 0;
    if (x0 < w) {
        const uint16_t *col = fr + x0;
        const bool vec = x0 + kSumPerThread <= w && (pitch & 7) == 0 && (reinterpret_cast<uintptr_t>(col) & 15) == 0;
        if (vec) {
            int y = blockIdx.y;
            for (; y + 3 * gy < h; y += 4 * gy) {
                const uint4 a = __ldg(reinterpret_cast<const uint4 *>(col + (size_t)y * pitch));
                const uint4 b = __ldg(reinterpret_cast<const uint4 *>(col + (size_t)(y + gy) * pitch));
                const uint4 c = __ldg(reinterpret_cast<const uint4 *>(col + (size_t)(y + 2 * gy) * pitch));
                const uint4 d = __ldg(reinterpret_cast<const uint4 *>(col + (size_t)(y + 3 * gy) * pitch));
                acc += (unsigned long long)sum8(a) + sum8(b) + sum8(c) + sum8(d);
            }
            for (; y < h; y += gy) acc += sum8(__ldg(reinterpret_cast<const uint4 *>(col + (size_t)y * pitch)));
        } else {
            for (int y = blockIdx.y; y < h; y += gy)
                for (int i = 0; i < kSumPerThread && x0 + i < w; ++i) acc += __ldg(col + (size_t)y * pitch + i);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0 && acc) atomicAdd(sum, acc);
}

// ---------------------------------------------------------------------------------------
// Monte-Carlo noise statistics (Sec. 5.2.2: sigma_md and d_md from simulations "for
// different brightness levels", with sensor clipping)
// ---------------------------------------------------------------------------------------
// a cluster of 8 blocks per brightness level: 1032 blocks of 4 warps, one wave at 7 blocks per
// SM (one block per level left 23 of 152 SMs idle and 8 warps on each of the others)
constexpr int kNoiseThreads = 128, kNoiseCluster = 8;
static_assert(kNoiseTrials % (kNoiseThreads * kNoiseCluster) == 0, "every thread takes the same number of trials");

// Philox-4x32-10 (Salmon et al., SC 2011): ten rounds of two 32x32 -> 64-bit products by
// fixed multipliers, the halves recombined with the other counter words and the round
// key; the key is bumped by the Weyl constants between rounds
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}

// normal j of a trial: 12 uniforms (r + 1/2) 2^-32 from three Philox blocks, summed exactly
// (Irwin-Hall), minus 6
__device__ __forceinline__ uint4 noise_block(int level, int trial, int j, int b) {
    return philox4x32_10(make_uint4((uint32_t)(3 * j + b), (uint32_t)trial, (uint32_t)level, 0u), 0x19050327u, 0x5EED0001u);
}

// one raw sample of a constant patch: rounded to a whole DN and clipped to [0, WL], in
// FP64 with the same operation sequence as a CPU restatement, so every decision agrees
__device__ __noinline__ int noise_sample_exact(double x, double sigma, int wl, int level, int trial, int j) {
    unsigned long long s = 0;
    for (int b = 0; b < 3; ++b) {
        const uint4 o = noise_block(level, trial, j, b);
        s += (unsigned long long)o.x + o.y + o.z + o.w;
    }
    const double z = __dadd_rn(__dmul_rn(__dadd_rn((double)s, 6.0), 1.0 / 4294967296.0), -6.0);
    const double v = floor(__dadd_rn(__dadd_rn(x, __dmul_rn(sigma, z)), 0.5));
    return (int)fmin(fmax(v, 0.0), (double)wl);
}

// One level's constants.  xi, xh: the brightness x as a whole number plus xh - 1/2 (x is a
// multiple of 1/128, so both are exact).
struct NoiseLevel {
    double x, sigma;
    float xh, sf, eb;
    int xi, wl, level;
};

// The same sample, decided in FP32: floor(xh + sigma z) with z from the uniforms' top 28 bits.
// Their truncation (12 x 16 x 2^-32 = 4.5e-8), the conversion and the two roundings are below
// 4e-7 |w| + 2e-7 sigma + 1e-6 of w; only a w closer than that to a whole number (1 sample in
// 10^4) takes the FP64 sequence, which this GPU issues at 1/64 of the FP32 rate.  All 28.5 M
// samples in FP64: 863 us; now 259, bound by the Philox integer products.
__device__ __forceinline__ int noise_sample(const NoiseLevel &n, int trial, int j) {
    uint32_t s = 0;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const uint4 o = noise_block(n.level, trial, j, b);
        s += (o.x >> 4) + (o.y >> 4) + (o.z >> 4) + (o.w >> 4);  // 12 x 2^28 < 2^32
    }
    const float z = (float)(int)(s - (6u << 28)) * (1.f / 268435456.f);
    const float w = fmaf(n.sf, z, n.xh), fl = floorf(w), fr = w - fl;
    const float e = fmaf(4e-7f, fabsf(w), n.eb);
    if (fabsf(w) < 131072.f && !(fr >= e && fr <= 1.f - e)) return noise_sample_exact(n.x, n.sigma, n.wl, n.level, trial, j);
    return min(max(n.xi + (int)fminf(fmaxf(fl, -131072.f), 131072.f), 0), n.wl);
}

// A trial draws two independent 3x3 patches of guide pixels (red/blue: one sample; green: the
// mean of two).  The statistics of whole numbers are whole numbers over constants, so the level's
// sums are exact 64-bit integers whatever the order: population variance of patch 1, (9 sum v^2 -
// (sum v)^2) / 81, red/blue and green (of the doubled green guide, over 4); squared difference of
// the two patch means, (S1 - S2)^2 / 81, red/blue and green.
__global__ void __cluster_dims__(kNoiseCluster, 1, 1) __launch_bounds__(kNoiseThreads)
    k_noise_table(float noise_a, float noise_b, int wl, float4 *__restrict__ table) {
    namespace cg = cooperative_groups;
    __shared__ unsigned long long red[kNoiseThreads / 32][4];
    NoiseLevel n;
    n.level = blockIdx.x / kNoiseCluster;
    n.wl = wl;
    n.x = __ddiv_rn(__dmul_rn((double)n.level, (double)wl), (double)(kNoiseLevels - 1));
    const double var = __dadd_rn(__dmul_rn((double)noise_a, n.x), (double)noise_b);
    n.sigma = var > 0.0 ? __dsqrt_rn(var) : 0.0;
    n.xi = (int)n.x;
    n.xh = (float)(n.x - (double)n.xi) + 0.5f;
    n.sf = (float)n.sigma;
    n.eb = fmaf(2e-7f, n.sf, 1e-6f);
    unsigned long long acc[4] = {0, 0, 0, 0};
    constexpr int kPer = kNoiseTrials / (kNoiseThreads * kNoiseCluster);
    const int t0 = (blockIdx.x % kNoiseCluster) * kNoiseThreads + threadIdx.x;
#pragma unroll 1
    for (int i = 0; i < kPer; ++i) {
        const int t = t0 + i * kNoiseThreads * kNoiseCluster;
        long long sum[2][2];  // [patch][red/blue, green]
#pragma unroll 1
        for (int q = 0; q < 2; ++q) {
            long long srb = 0, sg = 0;
            unsigned long long qrb = 0, qg = 0;
#pragma unroll 1
            for (int k = 0; k < 9; ++k) {
                const int v = noise_sample(n, t, 27 * q + k);
                const int gr = noise_sample(n, t, 27 * q + 9 + 2 * k) + noise_sample(n, t, 27 * q + 10 + 2 * k);
                srb += v;
                sg += gr;
                qrb += (unsigned long long)((long long)v * v);
                qg += (unsigned long long)((long long)gr * gr);
            }
            if (q == 0) {
                acc[0] += 9ull * qrb - (unsigned long long)(srb * srb);
                acc[1] += 9ull * qg - (unsigned long long)(sg * sg);
                sum[0][0] = srb; sum[0][1] = sg;
            } else {
                sum[1][0] = srb; sum[1][1] = sg;
            }
        }
        const long long d0 = sum[0][0] - sum[1][0], d1 = sum[0][1] - sum[1][1];
        acc[2] += (unsigned long long)(d0 * d0);
        acc[3] += (unsigned long long)(d1 * d1);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][k] = acc[k];
    }
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    if (cluster.block_rank() == 0 && threadIdx.x < 4) {
        unsigned long long s = 0;
        for (int r = 0; r < kNoiseCluster; ++r) {
            const unsigned long long *other = cluster.map_shared_rank(&red[0][0], r);
            for (int w = 0; w < kNoiseThreads / 32; ++w) s += other[w * 4 + threadIdx.x];
        }
        const double scale = 81.0 * kNoiseTrials * ((threadIdx.x & 1) ? 4.0 : 1.0);
        reinterpret_cast<float *>(table + n.level)[threadIdx.x] = (float)((double)s / scale);
    }
    cluster.sync();  // the other blocks' shared memory stays until it has been read
}

// piecewise-linear parameter between its value at SNR 6 (low) and at SNR 30 (high)
double lerp_snr(double lo, double hi, double snr) {
    const double t = fmin(fmax((snr - 6.0) / 24.0, 0.0), 1.0);
    return (1.0 - t) * lo + t * hi;  // both ends exact
}

}  // namespace
}  // namespace hmfsr

using namespace hmfsr;

extern "C" {

hmfsr_status hmfsr_frame_sum(const uint16_t *burst_dev, const hmfsr_burst_desc *desc, int frame,
                             unsigned long long *sum_dev, void *stream) {
    if (!desc || !burst_dev || !sum_dev || frame < 0 || frame >= desc->n_frames || desc->height < 1 ||
        desc->width < 1 || desc->pitch_elems < desc->width || (reinterpret_cast<uintptr_t>(sum_dev) & 7))
        return HMFSR_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (cudaMemsetAsync(sum_dev, 0, sizeof(unsigned long long), s) != cudaSuccess) return HMFSR_ERR_CUDA;
    const int gx = div_up(desc->width, kSumThreads * kSumPerThread);
    // about 4 blocks per SM in all, each thread over ~h / gy rows
    const int gy = max(1, min(div_up(desc->height, 4), (152 * 4) / gx));
    const uint16_t *fr = burst_dev + (size_t)frame * desc->height * desc->pitch_elems;
    k_frame_sum<<<dim3(gx, gy), kSumThreads, 0, s>>>(fr, desc->height, desc->width, desc->pitch_elems, sum_dev);
    return cudaGetLastError() == cudaSuccess ? HMFSR_OK : HMFSR_ERR_CUDA;
}

hmfsr_status hmfsr_noise_table(float noise_a, float noise_b, int white_level, float *table_dev, void *stream) {
    if (!table_dev || (reinterpret_cast<uintptr_t>(table_dev) & 15) || !isfinite(noise_a) || !isfinite(noise_b) ||
        noise_a < 0.f || noise_b < 0.f || white_level < 1 || white_level > 65535)
        return HMFSR_ERR_INVALID_ARG;
    k_noise_table<<<kNoiseLevels * kNoiseCluster, kNoiseThreads, 0, (cudaStream_t)stream>>>(noise_a, noise_b, white_level,
                                                                          reinterpret_cast<float4 *>(table_dev));
    return cudaGetLastError() == cudaSuccess ? HMFSR_OK : HMFSR_ERR_CUDA;
}

hmfsr_status hmfsr_snr_tuning(uint64_t sample_sum, uint64_t sample_count, float noise_a, float noise_b,
                              hmfsr_merge_params *mparams, hmfsr_align_params *aparams, double *snr_out) {
    // both below 2^53: exact as doubles, so the mean is the correctly rounded quotient
    if (!mparams || !aparams || sample_count == 0 || sample_count >= (1ull << 53) || sample_sum >= (1ull << 53) ||
        !isfinite(noise_a) || !isfinite(noise_b) || noise_a < 0.f || noise_b < 0.f)
        return HMFSR_ERR_INVALID_ARG;
    const double mean = (double)sample_sum / (double)sample_count;
    // SNR of one raw sample of a single frame at the mean brightness
    const double var = (double)noise_a * mean + (double)noise_b;
    const double snr = var > 0.0 ? mean / sqrt(var) : INFINITY;
    const double snr_c = isinf(snr) ? 30.0 : snr;
    // the tile grows from 16 px to 64 px only in very low light: the lowest third of the
    // SNR range, split in two
    const int tile = snr_c < 10.0 ? 64 : (snr_c < 14.0 ? 32 : 16);
    mparams->k_detail = (float)lerp_snr(0.33, 0.25, snr_c);
    mparams->k_denoise = (float)lerp_snr(5.0, 3.0, snr_c);
    mparams->d_th = (float)lerp_snr(0.010, 0.001, snr_c);
    mparams->d_tr = (float)lerp_snr(0.020, 0.006, snr_c);
    mparams->k_stretch = 4.f;
    mparams->k_shrink = 2.f;
    mparams->t = 0.12f;
    mparams->s1 = 12.f;
    mparams->s2 = 2.f;
    mparams->m_th = 0.8f;
    mparams->noise_a = noise_a;
    mparams->noise_b = noise_b;
    mparams->tile = tile;
    aparams->tile = tile;
    aparams->n_levels = 4;
    aparams->radius[0] = 1;
    aparams->radius[1] = aparams->radius[2] = aparams->radius[3] = 4;
    aparams->lk_iters = 3;
    if (snr_out) *snr_out = snr;
    return HMFSR_OK;
}

}  // extern "C"
