// The accumulation (Eq. 1-2) at scales 1, 3/2 and 2 with motion tiles of 16 px and more: one
// region of 16 x 16 raw pixels (8 x 8 half-res texels, inside one motion tile) per thread block.
//
// Why regions.  A region's output pixels share each frame's motion, and at these scales a whole
// number S of output pixels covers a half-res texel, so the S x S pixels of every texel have the
// same S x S phases against the Omega and Bayer grids.  A warp takes one phase: window offsets,
// their squares, Omega's bilinear weights and the window's Bayer arrangement are the same for all
// its lanes and come from a small table made once per region and frame (AxisTab); the Bayer
// arrangement is a uniform branch instead of selects per sample.  A lane's two pixels (the same
// phase of texels (u, v) and (u, v + 1)) run in packed FP32 pairs (fma.rn.f32x2: two IEEE
// operations per issue slot, bits as scalar).  A region's texels, raw samples and Rhat are staged
// in shared memory a frame ahead, and the squared cross products of det(Omega) (omega_form) are
// formed once per texel cell instead of once per pixel.
//
// What bounds it: issue and shared-memory bandwidth, 12 MP x 8 at scale 1: 244 warp-instructions
// per 32 pixel-frames (the 2 x 2-pixel kernel it replaces: 271), issue 68 %, shared-memory data
// path 77 %; DRAM 0.9 TB/s; 882 us (ncu).  Calls of hmfsr_merge_accumulate (CUDA events), with the
// per-pixel kernels and now:
//   12 MP x 8, 1x    1147 -> 908 us      12 MP x 8, 1.5x   2756 -> 1964 us
//   12 MP x 15, 2x   8568 -> 5342 us     0.07 MP x 8, 1x     57 -> 33 us
#pragma once

#include <limits.h>

#include "accumulate.cuh"

namespace hmfsr {
namespace stage {

struct PairAcc {
    float2 numR, numG, numB, denR, denG, denB, mR, mG, mB;
};
__device__ __forceinline__ PixelAcc half_of(const PairAcc &a, bool hi) {
    PixelAcc p;
    p.numR = hi ? a.numR.y : a.numR.x; p.numG = hi ? a.numG.y : a.numG.x; p.numB = hi ? a.numB.y : a.numB.x;
    p.denR = hi ? a.denR.y : a.denR.x; p.denG = hi ? a.denG.y : a.denG.x; p.denB = hi ? a.denB.y : a.denB.x;
    p.mR = hi ? a.mR.y : a.mR.x; p.mG = hi ? a.mG.y : a.mG.x; p.mB = hi ? a.mB.y : a.mB.x;
    return p;
}
__device__ __forceinline__ PairAcc join_halves(const PixelAcc &a, const PixelAcc &b) {
    PairAcc p;
    p.numR = make_float2(a.numR, b.numR); p.numG = make_float2(a.numG, b.numG); p.numB = make_float2(a.numB, b.numB);
    p.denR = make_float2(a.denR, b.denR); p.denG = make_float2(a.denG, b.denG); p.denB = make_float2(a.denB, b.denB);
    p.mR = make_float2(a.mR, b.mR); p.mG = make_float2(a.mG, b.mG); p.mB = make_float2(a.mB, b.mB);
    return p;
}


constexpr float kTop = 96.f;    // largest exponent of a weight: sums of 4096 frames x 9 samples below 2^13 stay finite
constexpr int kTexN = 11;   // staged texels per axis: cells -1 .. 8 of 8 texels, one more to interpolate
constexpr int kTexP = 12;   // pitch of the staged planes of single words (8 x 4 lanes, two rows apart: no bank conflicts)
constexpr int kRawP = 18;   // pitch of a staged raw row's even (or odd) samples
constexpr int kRawH = 2 * kTexN;
constexpr int kRawOdd = kRawH * kRawP;  // the odd samples' plane follows the even one's
constexpr int kRing = 8;                // frames whose constants are held

// One frame's constants of one phase along one axis, pairs doubled for the packed operations
struct AxisTab {
    float4 d01;   // {d-, d-, d0, d0}: offsets of the window's columns (rows) from the sampling point
    float4 d2s0;  // {d+, d+, d-^2, d-^2}
    float4 s12;   // {d0^2, d0^2, d+^2, d+^2}
    float4 fr;    // {1-f, 1-f, f, f}: Omega's bilinear fraction
    float4 q;     // {f (1-f), (1-f)^2, f^2, bits: cell offset | hi << 8 | border << 9}
};

template <int S>
struct RegionSmem {
    struct Frame {
        float4 om[kTexN * kTexN];  // {a, delta uy^2, -2 delta ux uy, delta ux^2}
        // det(M) terms: edge to the right, edge downwards, the cell's two diagonals (planes of
        // single words, which 8 x 4 lanes of texel pairs read without bank conflicts)
        float ch[kTexN * kTexP], cv[kTexN * kTexP], cd[kTexN * kTexP];
        float rh[kTexN * kTexP];   // Rhat texels
        float raw[2 * kRawOdd];    // raw samples: even columns, then odd ones
    } fr[2];
    float4 tex[2][(kTexN + 1) * kTexN + 1];  // staged texels {a, delta, ux, uy}; one row past the end is read, never used
    AxisTab tab[kRing][2 * S];           // x phases, then y phases
    struct Desc {
        const float4 *tex;    // the frame's first staged texel and raw sample
        const uint16_t *raw;
        const float *rh;
        int cx, cy;           // first staged texel; cx = kBorder: not wholly inside the frame
    } desc[kRing];
};

// asynchronous copies into shared memory (plain checked accesses in the checked build)
__device__ __forceinline__ void copy16(float4 *dst, const float4 *src) {
#ifdef HMFSR_CHECKED
    *dst = HMFSR_LDG(src);
#else
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
#endif
}
__device__ __forceinline__ void copy4(float *dst, const float *src) {
#ifdef HMFSR_CHECKED
    *dst = HMFSR_LDG(src);
#else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
#endif
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// keeps a value that a loop uses in its register: without it the compiler derives it again
// (index divisions, clamps) in every iteration to save the register
__device__ __forceinline__ void keep(int &x) { asm volatile("" : "+r"(x)); }
__device__ __forceinline__ void keep(float &x) { asm volatile("" : "+f"(x)); }

template <int SN, int SD>
struct RegionScale {
    static_assert(2 * SN % SD == 0, "a whole number of output pixels per half-res pixel");
    static constexpr int S = 2 * SN / SD;        // output pixels per half-res pixel
    static constexpr int kOff = S > 2 ? 1 : 0;   // first output pixel at or after raw position 0
};
// which scales take regions: 1 (1/1), 2 (3/2) or 3 (2/1); 0: merge_px / merge_quad1.  A tile of
// 8 px would leave three quarters of a region's lanes idle.
__host__ __device__ __forceinline__ int region_kind(int tile, int num, int den) {
    if (tile < 16) return 0;
    return num == den ? 1 : (2 * num == 3 * den ? 2 : (num == 2 * den ? 3 : 0));
}
// Q of the window geometry (geo_entry): 2 x the scale's numerator in lowest terms for these
__host__ __device__ __forceinline__ int geo_q(int tile, int num, int den) {
    const int kind = region_kind(tile, num, den);
    return kind == 2 ? 6 : (kind == 3 ? 4 : (num == den ? 2 : 2 * num));
}
// regions along one axis
template <int SN, int SD>
__host__ __device__ __forceinline__ int region_count(int raw) {
    return div_up(raw, 16) + RegionScale<SN, SD>::kOff;  // one more where an output pixel lies before raw position 0
}
// (phases, texel pair) items of a region, NPX x phases to an item
template <int SN, int SD, int NPX>
__host__ __device__ constexpr int region_items() {
    return 32 * RegionScale<SN, SD>::S * (RegionScale<SN, SD>::S / NPX);
}

// cell (-1 or 0, relative to the texel) and phase in [0, 2Q) of a texel's output pixel s at F = 0
template <int SN, int SD>
__device__ __forceinline__ int region_phase(int s, int &c) {
    const int P = 2 * SD * (RegionScale<SN, SD>::kOff + s) + SD - 2 * SN;
    c = P < 0 ? -1 : 0;
    return P < 0 ? P + 4 * SN : P;
}

// The staging of a region's frames in shared memory by the NT threads of a block.  Who stages
// what: texels the first 121 threads, Rhat and the cross products the next warps where there are
// enough, raw words from the last thread down.
// kHold: a thread's raw samples wait for their turn in registers, else in shared memory as they are
template <int SN, int SD, int NT, bool kHold>
struct RegionStage {
    static constexpr int S = RegionScale<SN, SD>::S, kOff = RegionScale<SN, SD>::kOff;
    static constexpr int Q = 2 * SN, Q2 = 4 * SN;
    static constexpr int kTexT = kTexN * kTexN, kRawT = kTexN * kRawH;
    static constexpr int kRawL = (kRawT + NT - 1) / NT, kTexL = (kTexT + NT - 1) / NT, kNext = NT >= 256 ? 128 : 0;
    using Smem = RegionSmem<S>;
    Smem &sm;
    const uint16_t *burst;
    const int4 *geo_r;
    const Geom &g;
    const float4 *kern;
    const float *rhat_planes;
    int U0, V0, tid;
    int tso[kTexL], tgo[kTexL], rgo[kTexL], cso[kTexL], wso[kRawL], wgo[kRawL];
    uint32_t held[kHold ? kRawL : 1];

    __device__ __forceinline__ RegionStage(Smem &sm_, const uint16_t *burst_, const int4 *geo, const Geom &g_,
                                           const float4 *kern_, const float *rhat_, int bx, int by, int tid_)
        : sm(sm_), burst(burst_), g(g_), kern(kern_), rhat_planes(rhat_), U0((bx - kOff) * 8), V0((by - kOff) * 8),
          tid(tid_) {
        geo_r = geo + (size_t)clampi(2 * V0 / g.tile, 0, g.ty - 1) * g.tx + clampi(2 * U0 / g.tile, 0, g.tx - 1);
#pragma unroll
        for (int k = 0; k < kTexL; ++k) {
            const int i = tid + k * NT, r = i / kTexN, c = i - r * kTexN;
            tso[k] = i < kTexT ? i : -1;
            tgo[k] = r * g.wh + c;
            const int j = i - kNext, rr = j / kTexN, rc = j - rr * kTexN;
            rgo[k] = clampi(V0 - 1 + rr, 0, g.hh - 1) * g.wh + clampi(U0 - 1 + rc, 0, g.wh - 1);
            cso[k] = j >= 0 && j < kTexT ? j | (rr * kTexP + rc) << 8 : -1;  // texel | index in the planes << 8
            keep(tso[k]); keep(tgo[k]); keep(rgo[k]); keep(cso[k]);
        }
#pragma unroll
        for (int k = 0; k < kRawL; ++k) {
            const int i = NT - 1 - tid + k * NT, r = i / kTexN, c = i - r * kTexN;
            wso[k] = i < kRawT ? r * kRawP + c : -1;
            wgo[k] = r * g.pitch + 2 * c;
            keep(wso[k]); keep(wgo[k]);
        }
    }
    // the constants of frames [first, first + count) of the accumulation order
    __device__ __forceinline__ void fill(int first, int count) {
        constexpr float invQ = 1.f / (float)Q, inv2Q = 0.5f / (float)Q;
        const size_t hw = (size_t)g.hh * g.wh, ntl = (size_t)g.ty * g.tx, fstride = (size_t)g.h * g.pitch;
        for (int i = tid; i < count * 2 * S; i += NT) {
            const int it = first + i / (2 * S), k = i % (2 * S), f = frame_of_step(it, g.ref);
            const int4 e = HMFSR_LDG(geo_r + (size_t)f * ntl);
            const int cx = U0 - 1 + (e.x >> 6), cy = V0 - 1 + (e.y >> 6);
            const bool in = cx >= 0 && cx + kTexN <= g.wh && cy >= 0 && cy + kTexN <= g.hh;
            const bool isy = k >= S;
            const float z = __int_as_float(isy ? e.w : e.z);
            int c;
            int p = region_phase<SN, SD>(isy ? k - S : k, c) + ((isy ? e.y : e.x) & 63);
            if (p >= Q2) { p -= Q2; ++c; }
            const bool hi = p >= Q;
            const float d0 = ((float)(SN - p + (hi ? Q : 0)) - z) * invQ, dm = d0 - 1.f, dp = d0 + 1.f;
            const float fr = ((float)p + z) * inv2Q, f1 = 1.f - fr;
            AxisTab &a = sm.tab[it & (kRing - 1)][k];
            a.d01 = make_float4(dm, dm, d0, d0);
            a.d2s0 = make_float4(dp, dp, dm * dm, dm * dm);
            a.s12 = make_float4(d0 * d0, d0 * d0, dp * dp, dp * dp);
            a.fr = make_float4(f1, f1, fr, fr);
            a.q = make_float4(fr * f1, f1 * f1, fr * fr,
                              __int_as_float((c + 1) | (hi ? 256 : 0) | (in ? 0 : 512)));
            if (k == 0) {
                typename Smem::Desc &d = sm.desc[it & (kRing - 1)];
                const ptrdiff_t o = (ptrdiff_t)f * (ptrdiff_t)hw;
                d.tex = kern + o + (in ? (ptrdiff_t)cy * g.wh + cx : 0);
                d.raw = burst + (size_t)src_frame(g, f) * fstride + (in ? (ptrdiff_t)2 * cy * g.pitch + 2 * cx : 0);
                d.rh = rhat_planes + o;
                d.cx = in ? INT_MIN : cx;
                d.cy = cy;
            }
        }
    }
    __device__ __forceinline__ const typename Smem::Desc &desc(int it) const { return sm.desc[it & (kRing - 1)]; }
    __device__ __forceinline__ void stage_tex(float4 *dst, int it) {
        const typename Smem::Desc &d = desc(it);
        if (d.cx == INT_MIN) {
            const float4 *p = d.tex;
#pragma unroll
            for (int k = 0; k < kTexL; ++k)
                if (tso[k] >= 0) copy16(dst + tso[k], p + tgo[k]);
        } else {
            for (int i = tid; i < kTexT; i += NT) {
                const int r = i / kTexN, c = i - r * kTexN;
                copy16(dst + i, d.tex + (clampi(d.cy + r, 0, g.hh - 1) * g.wh + clampi(d.cx + c, 0, g.wh - 1)));
            }
        }
    }
    __device__ __forceinline__ void stage_rhat(float *dst, int it) {
        if (it == 0) return;  // the base frame
        const float *p = desc(it).rh;
#pragma unroll
        for (int k = 0; k < kTexL; ++k)
            if (cso[k] >= 0) copy4(dst + (cso[k] >> 8), p + rgo[k]);
    }
    // pairs of raw samples, as they are, into registers or the even plane; spread_raw turns a thread's
    // own pairs into the two planes once they have arrived.  Registers cost less at the shared-memory
    // path (merging at scale 1, which that path bounds: 1.6 % of the call at 12 MP x 8), shared
    // memory where registers are short (3/2: 0.7 %; the adjoint, which spilled).
    __device__ __forceinline__ void stage_raw(float *dst, int it) {
        const typename Smem::Desc &d = desc(it);
        const uint16_t *p = d.raw;
        if (d.cx == INT_MIN) {
#pragma unroll
            for (int k = 0; k < kRawL; ++k)
                if (wso[k] >= 0) {
                    if (kHold) held[k] = HMFSR_LDG(reinterpret_cast<const uint32_t *>(p + wgo[k]));
                    else copy4(dst + wso[k], reinterpret_cast<const float *>(p + wgo[k]));
                }
        } else {
#pragma unroll
            for (int k = 0; k < kRawL; ++k) {
                const int i = NT - 1 - tid + k * NT, r = i / kTexN, c = i - r * kTexN;
                const uint16_t *q = p + (clampi(2 * d.cy + r, 0, g.h - 1) * g.pitch + 2 * clampi(d.cx + c, 0, g.wh - 1));
                if (i < kRawT) {
                    if (kHold) held[k] = HMFSR_LDG(reinterpret_cast<const uint32_t *>(q));
                    else copy4(dst + wso[k], reinterpret_cast<const float *>(q));
                }
            }
        }
    }
    __device__ __forceinline__ void spread_raw(float *dst) {
#pragma unroll
        for (int k = 0; k < kRawL; ++k)
            if (wso[k] >= 0) {
                const uint32_t w = kHold ? held[k] : __float_as_uint(dst[wso[k]]);
                dst[wso[k]] = (float)(w & 0xffffu);
                dst[kRawOdd + wso[k]] = (float)(w >> 16);
            }
    }
    // per texel M = delta u u^T, per cell the squared cross products
    __device__ __forceinline__ void derive(int b) {
#pragma unroll
        for (int k = 0; k < kTexL; ++k) {
            if (cso[k] >= 0) {
                const float4 *T = sm.tex[b] + (cso[k] & 255);
                const float4 t0 = T[0], t1 = T[1], t2 = T[kTexN], t3 = T[kTexN + 1];
                auto cross = [](const float4 &s, const float4 &t) {
                    const float w = fmaf(s.z, t.w, -(s.w * t.z));
                    return (s.y * w) * (t.y * w);
                };
                const int o = cso[k] >> 8;
                sm.fr[b].ch[o] = cross(t0, t1);
                sm.fr[b].cv[o] = cross(t0, t2);
                sm.fr[b].cd[o] = cross(t0, t3) + cross(t1, t2);
            }
            if (tso[k] >= 0) {
                const float4 t0 = sm.tex[b][tso[k]];
                const float my = t0.y * t0.w;
                sm.fr[b].om[tso[k]] = make_float4(t0.x, my * t0.w, -2.f * (my * t0.z), t0.y * t0.z * t0.z);
            }
        }
    }
    // the first frame whole, the second's texels
    __device__ __forceinline__ void begin(int it0) {
        fill(it0, min(kRing, g.n - it0));
        __syncthreads();
        stage_tex(sm.tex[it0 & 1], it0);
        stage_rhat(sm.fr[it0 & 1].rh, it0);
        stage_raw(sm.fr[it0 & 1].raw, it0);
        if (it0 + 1 < g.n) stage_tex(sm.tex[(it0 + 1) & 1], it0 + 1);
        copy_wait();
        spread_raw(sm.fr[it0 & 1].raw);
        __syncthreads();
        derive(it0 & 1);
        __syncthreads();
    }
    // while frame `it` is worked on (and the constants of kLag frames before it may still be read):
    // the next frame's copies and derived terms
    template <int kLag = 0>
    __device__ __forceinline__ void ahead(int it, int it0) {
        const int b = it & 1;
        if (it + 1 >= g.n) return;
        stage_raw(sm.fr[b ^ 1].raw, it + 1);
        stage_rhat(sm.fr[b ^ 1].rh, it + 1);
        if (it + 2 < g.n) stage_tex(sm.tex[b], it + 2);
        derive(b ^ 1);
        // frames up to it + 2 are in use, and from it - kLag on: the slots half a ring on are free
        constexpr int kBatch = kRing / 2 - kLag;
        static_assert((kBatch & (kBatch - 1)) == 0 && kRing / 2 >= 4, "a batch ends before frame it - kLag's slot");
        const int next = it + kRing / 2;
        if (next >= it0 + kRing && (it - it0) % kBatch == 0 && next < g.n) fill(next, min(kBatch, g.n - next));
    }
    // after it: the raw samples into place, and the block in step
    __device__ __forceinline__ void advance(int it) {
        if (it + 1 >= g.n) return;
        copy_wait();
        spread_raw(sm.fr[(it & 1) ^ 1].raw);
        __syncthreads();
    }
};

// Items [item0, item0 + NT) of region (bx, by), all frames.  Every thread of the block calls this.
// NPX x phases per thread share their Omega cell and window where they fall on the same ones
// (fewer shared-memory reads, more registers); the results do not depend on it.
template <bool kDen, int SN, int SD, int NT, int NPX, bool kChunk = false>
__device__ __forceinline__ void merge_region(RegionSmem<RegionScale<SN, SD>::S> &sm, const uint16_t *__restrict__ burst,
                                             const int4 *__restrict__ geo, const Geom &g,
                                             const float4 *__restrict__ kern, const float *__restrict__ rhat_planes,
                                             int ho, int wo, float *__restrict__ rgb, float *__restrict__ den_out,
                                             int bx, int by, int item0, int tid, const ChunkIO &io = ChunkIO{}) {
    constexpr int S = RegionScale<SN, SD>::S, kOff = RegionScale<SN, SD>::kOff;
    constexpr float inv2Q = 0.25f / (float)SN;
    const int U0 = (bx - kOff) * 8, V0 = (by - kOff) * 8;  // the region's first texel

    // this thread's pair: phases (sx, sy) of texels (u, v) and (u, v + 1) of the region
    const int item = item0 + tid, pr = item & 31, phase = item >> 5;
    const int sy = phase / (S / NPX), sx = (phase - sy * (S / NPX)) * NPX;  // phases sx .. sx + NPX - 1
    const int v = 2 * (pr >> 3), u = pr & 7;
    const int X = S * (U0 + u) + kOff + sx, Y = S * (V0 + v) + kOff + sy;
    auto valid = [&](int k, int h) { return sy < S && X + k >= 0 && X + k < wo && Y + h * S >= 0 && Y + h * S < ho; };
    const bool active = sy < S && X + NPX > 0 && X < wo && Y + S >= 0 && Y < ho;
    RegionStage<SN, SD, NT, SN == SD> st(sm, burst, geo, g, kern, rhat_planes, bx, by, tid);

    PixelAcc none;
    none.mR = none.mG = none.mB = 0.f;  // the first frame's exponents are -q'; it then sets the shifts
    PairAcc acc[NPX];
    int it0 = 0;
    bool fresh = true;
#pragma unroll
    for (int k = 0; k < NPX; ++k) acc[k] = join_halves(none, none);
    if constexpr (kChunk) {
        it0 = io.skip_base ? 1 : 0;
        if (io.state_in) {
            fresh = false;
#pragma unroll
            for (int k = 0; k < NPX; ++k) {
                PixelAcc s0, s1;
                if (valid(k, 0)) load_state(io, (size_t)Y * wo + X + k, s0);
                if (valid(k, 1)) load_state(io, (size_t)(Y + S) * wo + X + k, s1);
                acc[k] = join_halves(s0, s1);
            }
        }
    }
    // a sample's weight is 2^(m - q') with q' >= 0: while no shift m exceeds kTop none can overflow
    auto shifts_big = [&]() {
        float m = 0.f;
#pragma unroll
        for (int k = 0; k < NPX; ++k)
            m = fmaxf(m, fmaxf(fmaxf(fmaxf(acc[k].mR.x, acc[k].mR.y), fmaxf(acc[k].mG.x, acc[k].mG.y)),
                               fmaxf(acc[k].mB.x, acc[k].mB.y)));
        return !(m <= kTop);
    };
    bool big = fresh || shifts_big();
    float rfx[NPX], rfy;
    int ro[NPX], rcx, rcy;
    rfy = (float)region_phase<SN, SD>(sy, rcy) * inv2Q;
    keep(rfy);
#pragma unroll
    for (int k = 0; k < NPX; ++k) {
        rfx[k] = (float)region_phase<SN, SD>(sx + k, rcx) * inv2Q;
        ro[k] = (v + 1 + rcy) * kTexP + u + 1 + rcx;  // Rhat cell in shared memory
        keep(rfx[k]); keep(ro[k]);
    }
    int o0 = v * kTexP + u, m0 = v * kTexN + u, w0 = 2 * v * kRawP + u, txo = sx, tyo = S + sy, act = active ? 1 : 0;
    keep(o0); keep(m0); keep(w0); keep(txo); keep(tyo); keep(act);
    if (it0 < g.n) st.begin(it0);
    for (int it = it0; it < g.n; ++it) {
        const int b = it & 1;
        st.ahead(it, it0);
        do {  // left early where the frame adds nothing
            if (!act) break;
            const typename RegionSmem<S>::Frame &fr = sm.fr[b];
            float2 rh[NPX];
            bool any = it == 0;
#pragma unroll
            for (int k = 0; k < NPX; ++k) {
                rh[k] = make_float2(1.f, 1.f);
                if (it > 0) {
                    const float *R = fr.rh + ro[k];
                    const float rfx1 = 1.f - rfx[k], rfy1 = 1.f - rfy;
                    const float h0 = fmaf(rfx[k], R[1], rfx1 * R[0]), h1 = fmaf(rfx[k], R[kTexP + 1], rfx1 * R[kTexP]);
                    const float h2 = fmaf(rfx[k], R[2 * kTexP + 1], rfx1 * R[2 * kTexP]);
                    rh[k].x = fmaf(rfy, h1, rfy1 * h0);
                    rh[k].y = fmaf(rfy, h2, rfy1 * h1);
                    any |= rh[k].x > 0.f || rh[k].y > 0.f;
                }
            }
            if (!any) break;
            const AxisTab *tx = &sm.tab[it & (kRing - 1)][txo], &ty = sm.tab[it & (kRing - 1)][tyo];
            const float4 qy = ty.q;
            const int ky = __float_as_int(qy.w);
            const bool hiy = (ky & 256) != 0;
            // Omega at the pixels: along x for the three texel rows, then along y
            float2 nBx[NPX], nBy[NPX], nBxy[NPX];
            int kx[NPX];
            {
                float4 tl[3], tr[3];
                float ch[3], cl[2], cr[2], cd[2];
                const float4 fy = ty.fr;
#pragma unroll
                for (int k = 0; k < NPX; ++k) {
                    const float4 qx = tx[k].q, fx = tx[k].fr;
                    kx[k] = __float_as_int(qx.w);
                    const int o = o0 + (kx[k] & 255) + (ky & 255) * kTexP, m = m0 + (kx[k] & 255) + (ky & 255) * kTexN;
                    if (k == 0 || (kx[k] & 255) != (kx[k - 1] & 255)) {  // the same for the whole warp
#pragma unroll
                        for (int j = 0; j < 3; ++j) {
                            if (k == 0) {
                                tl[j] = fr.om[m + j * kTexN];
                            } else {
                                tl[j] = tr[j];  // the next cell's left column
                            }
                            tr[j] = fr.om[m + j * kTexN + 1];
                            ch[j] = fr.ch[o + j * kTexP];
                        }
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            cl[h] = k == 0 ? fr.cv[o + h * kTexP] : cr[h];
                            cr[h] = fr.cv[o + h * kTexP + 1];
                            cd[h] = fr.cd[o + h * kTexP];
                        }
                    }
                    float2 l[3], r[3];  // {a, Mxx}, {Mxy, Myy}
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        l[j] = fma2(hi2(fx), lo2(tr[j]), mul2(lo2(fx), lo2(tl[j])));
                        r[j] = fma2(hi2(fx), hi2(tr[j]), mul2(lo2(fx), hi2(tl[j])));
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float2 L = fma2(hi2(fy), l[h + 1], mul2(lo2(fy), l[h])), R = fma2(hi2(fy), r[h + 1], mul2(lo2(fy), r[h]));
                        const float u1 = fmaf(qy.z, ch[h + 1], qy.y * ch[h]);
                        const float u2 = fmaf(qx.x, cd[h], fmaf(qx.z, cr[h], qx.y * cl[h]));
                        const float dM = fmaf(qx.x, u1, qy.x * u2);
                        const float s1 = L.x + L.y;
                        const float det = fmaf(L.x, s1 + R.y, dM);
                        const float sc = -kHalfLog2e * fast_rcp(det);
                        const float vx = s1 * sc, vy = (L.x + R.y) * sc, vxy = R.x * sc;
                        if (h) { nBx[k].y = vx; nBy[k].y = vy; nBxy[k].y = vxy; }
                        else { nBx[k].x = vx; nBy[k].x = vy; nBxy[k].x = vxy; }
                    }
                }
            }
            const float4 dya = ty.d01, dyb = ty.d2s0, dyc = ty.s12;
            const float2 dy[3] = {lo2(dya), hi2(dya), lo2(dyb)}, yy[3] = {hi2(dyb), lo2(dyc), hi2(dyc)};
            const bool first = fresh && it == it0;
            float col[3][5];  // raw columns of the windows
            const float *W = fr.raw + (w0 + 2 * kRawP * (ky & 255) + (hiy ? kRawP : 0));
            auto load_cols = [&](int ofs, bool hix) {
                const float *Wa = W + ofs + (hix ? kRawOdd : 0), *Wb = W + ofs + (hix ? 1 : kRawOdd);
#pragma unroll
                for (int j = 0; j < 5; ++j) {
                    col[0][j] = Wa[j * kRawP];
                    col[1][j] = Wb[j * kRawP];
                    col[2][j] = Wa[j * kRawP + 1];
                }
            };
#pragma unroll
            for (int k = 0; k < NPX; ++k) {
                const bool hix = (kx[k] & 256) != 0;
                PairAcc &a = acc[k];
                // exponents t = m - q' of the nine samples' weights
                const float4 dxa = tx[k].d01, dxb = tx[k].d2s0, dxc = tx[k].s12;
                const float2 xx[3] = {hi2(dxb), lo2(dxc), hi2(dxc)};
                const float2 be[3] = {mul2(nBxy[k], lo2(dxa)), mul2(nBxy[k], hi2(dxa)), mul2(nBxy[k], lo2(dxb))};
                float2 t[3][3];
                {
                    const float2 nb = nBy[k];
                    float2 r0K, r0V, r1H, r1C, r2K, r2V;  // shift of the class - Byy dy^2, per row
                    if (hix != hiy) {
                        r0K = fma2(nb, yy[0], a.mG); r2K = fma2(nb, yy[2], a.mG); r1C = fma2(nb, yy[1], a.mG);
                        if (hiy) {
                            r1H = fma2(nb, yy[1], a.mR); r0V = fma2(nb, yy[0], a.mB); r2V = fma2(nb, yy[2], a.mB);
                        } else {
                            r1H = fma2(nb, yy[1], a.mB); r0V = fma2(nb, yy[0], a.mR); r2V = fma2(nb, yy[2], a.mR);
                        }
                    } else {
                        r1H = fma2(nb, yy[1], a.mG); r0V = fma2(nb, yy[0], a.mG); r2V = fma2(nb, yy[2], a.mG);
                        if (hiy) {
                            r1C = fma2(nb, yy[1], a.mR); r0K = fma2(nb, yy[0], a.mB); r2K = fma2(nb, yy[2], a.mB);
                        } else {
                            r1C = fma2(nb, yy[1], a.mB); r0K = fma2(nb, yy[0], a.mR); r2K = fma2(nb, yy[2], a.mR);
                        }
                    }
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        t[0][i] = fma2(be[i], dy[0], fma2(nBx[k], xx[i], i == 1 ? r0V : r0K));
                        t[1][i] = fma2(be[i], dy[1], fma2(nBx[k], xx[i], i == 1 ? r1C : r1H));
                        t[2][i] = fma2(be[i], dy[2], fma2(nBx[k], xx[i], i == 1 ? r2V : r2K));
                    }
                }
                if (kx[k] & 512) {  // samples outside the frame are left out
                    const typename RegionSmem<S>::Desc &d = st.desc(it);
                    const int ax = 2 * (d.cx + u + (kx[k] & 255)) + (hix ? 1 : 0), ay = 2 * (d.cy + v + (ky & 255)) + (hiy ? 1 : 0);
#pragma unroll
                    for (int j = 0; j < 3; ++j)
#pragma unroll
                        for (int i = 0; i < 3; ++i) {
                            const bool xok = (unsigned)(ax + i) < (unsigned)g.w;
                            if (!(xok && (unsigned)(ay + j) < (unsigned)g.h)) t[j][i].x = -INFINITY;
                            if (!(xok && (unsigned)(ay + 2 + j) < (unsigned)g.h)) t[j][i].y = -INFINITY;
                        }
                }
                if (big) {
                    // a shift may have to be set (first frame: t = -q') or moved: a channel whose largest
                    // t is over kTop takes it off its shift and sums
                    const float2 xC = t[1][1];
                    const float2 xH = make_float2(fmaxf(t[1][0].x, t[1][2].x), fmaxf(t[1][0].y, t[1][2].y));
                    const float2 xV = make_float2(fmaxf(t[0][1].x, t[2][1].x), fmaxf(t[0][1].y, t[2][1].y));
                    const float2 xK = make_float2(fmaxf(fmaxf(t[0][0].x, t[0][2].x), fmaxf(t[2][0].x, t[2][2].x)),
                                                  fmaxf(fmaxf(t[0][0].y, t[0][2].y), fmaxf(t[2][0].y, t[2][2].y)));
                    const float ta = fmaxf(fmaxf(xC.x, xH.x), fmaxf(xV.x, xK.x)), tb = fmaxf(fmaxf(xC.y, xH.y), fmaxf(xV.y, xK.y));
                    if (first || !(ta <= kTop && tb <= kTop)) {
                        auto move = [&](float tmax, float rhv, float &m, float &num, float &den, float &d) {
                            d = 0.f;
                            if (!(rhv > 0.f)) return;
                            if (first) {
                                m = tmax == -INFINITY ? kBig : -tmax;
                                d = m;
                            } else if (tmax > kTop) {
                                const float s = fast_exp2(-tmax);
                                num *= s; den *= s;
                                d = -tmax;
                                m += d;
                            }
                        };
                        const bool cg = hix != hiy;
                        float2 dR, dG, dB;
                        const float2 tG = cg ? make_float2(fmaxf(xC.x, xK.x), fmaxf(xC.y, xK.y))
                                             : make_float2(fmaxf(xH.x, xV.x), fmaxf(xH.y, xV.y));
                        const float2 t1 = cg ? xH : xC, t2 = cg ? xV : xK;
                        const float2 tR = hiy ? t1 : t2, tB = hiy ? t2 : t1;
                        move(tR.x, rh[k].x, a.mR.x, a.numR.x, a.denR.x, dR.x);
                        move(tG.x, rh[k].x, a.mG.x, a.numG.x, a.denG.x, dG.x);
                        move(tB.x, rh[k].x, a.mB.x, a.numB.x, a.denB.x, dB.x);
                        move(tR.y, rh[k].y, a.mR.y, a.numR.y, a.denR.y, dR.y);
                        move(tG.y, rh[k].y, a.mG.y, a.numG.y, a.denG.y, dG.y);
                        move(tB.y, rh[k].y, a.mB.y, a.numB.y, a.denB.y, dB.y);
                        if (k == NPX - 1 || !first) big = shifts_big() || (first && k < NPX - 1);
                        const float2 dS1 = hiy ? dR : dB, dS2 = hiy ? dB : dR;
                        const float2 eC = cg ? dG : dS1, eK = cg ? dG : dS2, eH = cg ? dS1 : dG, eV = cg ? dS2 : dG;
#pragma unroll
                        for (int j = 0; j < 3; ++j)
#pragma unroll
                            for (int i = 0; i < 3; ++i) {
                                t[j][i] = add2(t[j][i], j == 1 ? (i == 1 ? eC : eH) : (i == 1 ? eV : eK));
                                if (!(rh[k].x > 0.f)) t[j][i].x = -INFINITY;  // a rejected frame adds nothing
                                if (!(rh[k].y > 0.f)) t[j][i].y = -INFINITY;
                            }
                    }
                }
                if (k == 0 || ((kx[k] ^ kx[k - 1]) & 511)) load_cols(kx[k] & 255, hix);  // pixels may share their window
                auto weight = [&](int j, int i) { return make_float2(fast_exp2(t[j][i].x), fast_exp2(t[j][i].y)); };
                auto value = [&](int j, int i) { return make_float2(col[i][j], col[i][j + 2]); };
                const float2 dC = weight(1, 1), nC = mul2(dC, value(1, 1));
                float2 wt = weight(1, 2);
                float2 dH = weight(1, 0), nH = mul2(dH, value(1, 0));
                nH = fma2(wt, value(1, 2), nH); dH = add2(dH, wt);
                wt = weight(2, 1);
                float2 dV = weight(0, 1), nV = mul2(dV, value(0, 1));
                nV = fma2(wt, value(2, 1), nV); dV = add2(dV, wt);
                float2 dK = weight(0, 0), nK = mul2(dK, value(0, 0));
                wt = weight(0, 2);
                nK = fma2(wt, value(0, 2), nK); dK = add2(dK, wt);
                wt = weight(2, 0);
                nK = fma2(wt, value(2, 0), nK); dK = add2(dK, wt);
                wt = weight(2, 2);
                nK = fma2(wt, value(2, 2), nK); dK = add2(dK, wt);
                // the window's classes onto the channels (the same for the whole warp)
                const float2 r = rh[k];
                if (hix != hiy) {
                    a.numG = fma2(r, add2(nC, nK), a.numG);
                    a.denG = fma2(r, add2(dC, dK), a.denG);
                    if (hiy) {
                        a.numR = fma2(r, nH, a.numR); a.denR = fma2(r, dH, a.denR);
                        a.numB = fma2(r, nV, a.numB); a.denB = fma2(r, dV, a.denB);
                    } else {
                        a.numR = fma2(r, nV, a.numR); a.denR = fma2(r, dV, a.denR);
                        a.numB = fma2(r, nH, a.numB); a.denB = fma2(r, dH, a.denB);
                    }
                } else {
                    a.numG = fma2(r, add2(nH, nV), a.numG);
                    a.denG = fma2(r, add2(dH, dV), a.denG);
                    if (hiy) {
                        a.numR = fma2(r, nC, a.numR); a.denR = fma2(r, dC, a.denR);
                        a.numB = fma2(r, nK, a.numB); a.denB = fma2(r, dK, a.denB);
                    } else {
                        a.numR = fma2(r, nK, a.numR); a.denR = fma2(r, dK, a.denR);
                        a.numB = fma2(r, nC, a.numB); a.denB = fma2(r, dC, a.denB);
                    }
                }
            }
        } while (false);
        st.advance(it);
    }
    const size_t po = (size_t)ho * wo;
#pragma unroll
    for (int k = 0; k < NPX; ++k)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (!valid(k, h)) continue;
            const PixelAcc p = half_of(acc[k], h);
            const size_t o = (size_t)(Y + h * S) * wo + X + k;
            if constexpr (kChunk) {
                if (io.state_out) {
                    store_state(io, o, p);
                    continue;
                }
            }
            HMFSR_ST(rgb + o, p.numR / p.denR);
            HMFSR_ST(rgb + po + o, p.numG / p.denG);
            HMFSR_ST(rgb + 2 * po + o, p.numB / p.denB);
            if (kDen) {
                HMFSR_ST(den_out + o, log2f(p.denR) - p.mR);
                HMFSR_ST(den_out + po + o, log2f(p.denG) - p.mG);
                HMFSR_ST(den_out + 2 * po + o, log2f(p.denB) - p.mB);
            }
        }
}

}  // namespace stage
}  // namespace hmfsr
