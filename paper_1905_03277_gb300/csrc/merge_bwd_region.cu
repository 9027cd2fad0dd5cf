// Adjoint of the merge by regions (scales 1, 3/2 and 2, motion tiles of 16 px and more): the
// forward's decomposition (accumulate_region.cuh) in reverse.  A block takes one region of a
// motion tile, a warp one phase of the output grid, a lane the two pixels of that phase on
// texels (u, v) and (u, v + 1), in packed FP32 pairs.
//
// What the per-pixel kernel (merge_bwd.cu, other scales and 8-px tiles) spends its 1145
// instructions per pixel-frame on, and where it goes here:
//   - window geometry by run-time division: from the region's table, once per frame;
//   - each of a pixel's four Omega texels through the kernel-shape derivatives: dL/dOmega is
//     linear, so it is first gathered onto the region's texels (the transposed bilinear
//     sampling, along x then y, in shared memory), and the derivatives run once per texel;
//   - motion contributions to a plane of pixels and back: summed in the block, which lies in one
//     tile; the R-hat contributions go out by phase, so that lanes write side by side and the
//     gather onto texels has constant weights.
// Fixed orders everywhere, so results are deterministic.
//
// Bounded by the issue rate (57 %) with the shared-memory path at 60 %: 659 warp-instructions per
// 32 pixel-frames.  At 1 MP x 8 frames, scale 3/2 (the fitting workload) the main kernel takes 550 us
// where the per-pixel one takes 802, the R-hat path 70 where its two kernels take 106.  Registers
// decide the rest: shared memory leaves little L1, so every word spilled in the frame loop goes to
// L2 (a version with 16 spilled words took 654 us).  Hence staging through shared memory and not
// registers, small blocks of one row of phases (3 warps, 5 blocks per SM; all nine phases in one
// block of 3 per SM, where 72 registers fit, took 726), and the constants re-derived.
#include "accumulate_region.cuh"
#include "adjoint_common.cuh"

namespace hmfsr {
namespace {

using stage::fma2;
using stage::mul2;
using stage::add2;
using stage::lo2;
using stage::hi2;
using stage::AxisTab;
using stage::kRing;
using stage::kTexN;
using stage::kTexP;
using stage::kRawP;
using stage::kRawOdd;
using stage::RegionScale;
using stage::RegionSmem;
using stage::RegionStage;

// kSy: y phases per block (the others go to further blocks, gridDim.z)
template <int SN, int SD>
struct AdjointShape;
template <> struct AdjointShape<1, 1> { static constexpr int kSy = 2, kBlocks = 4; };
template <> struct AdjointShape<3, 2> { static constexpr int kSy = 1, kBlocks = 5; };
template <> struct AdjointShape<2, 1> { static constexpr int kSy = 1, kBlocks = 4; };

constexpr int kObN = 100;        // a phase's 8 x 8 texels, rows of 12 with zeros around
constexpr int kObT = 14 * kTexP; // gathered along x: rows -3 .. 10 (zeros outside 0 .. 7)

// Motion contributions are summed times this (exactly): a warp's 64 pixels, or an 8 x 8 block's
// texels, cannot leave FP32's range together where each is inside it, and FP64 takes over from there
constexpr float kPart = 1.f / 64.f;

template <int S, int kSy>
struct AdjointSmem {
    RegionSmem<S> st;
    float2 px[kSy * S][9][32];  // per pixel pair: -log2 den, dL/dC and -dL/dC x C of R, G, B
    double red[kSy * S][12];
    float ob[2][kSy * S][3][kObN];
    float obx[2][kSy][3][kObT];
    float4 sh[2][kTexN * kTexN];
};

template <int SN, int SD>
__global__ void __launch_bounds__(32 * AdjointShape<SN, SD>::kSy *RegionScale<SN, SD>::S, AdjointShape<SN, SD>::kBlocks)
    k_adjoint_region(const uint16_t *__restrict__ burst, const int4 *__restrict__ geo, Geom g, MergeConsts c, KConsts kc,
                     const float4 *__restrict__ kern, const float4 *__restrict__ shape,
                     const float *__restrict__ rhat_planes, int ho, int wo, const float *__restrict__ rgb,
                     const float *__restrict__ lden, const float *__restrict__ grad_rgb,
                     float *__restrict__ rhbar_phase, float2 *__restrict__ vbar_region, double *__restrict__ partials) {
    constexpr int S = RegionScale<SN, SD>::S, kOff = RegionScale<SN, SD>::kOff, kSy = AdjointShape<SN, SD>::kSy;
    constexpr int NW = kSy * S, NT = 32 * NW;
    constexpr float inv2Q = 0.25f / (float)SN;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    AdjointSmem<S, kSy> &sm = *reinterpret_cast<AdjointSmem<S, kSy> *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int U0 = (blockIdx.x - kOff) * 8, V0 = (blockIdx.y - kOff) * 8;
    const int syl = warp / S, sy = blockIdx.z * kSy + syl, sx = warp - syl * S;
    const int v = 2 * (lane >> 3), u = lane & 7;
    const int X = S * (U0 + u) + kOff + sx, Y = S * (V0 + v) + kOff + sy;
    const size_t po = (size_t)ho * wo;
    for (int i = tid; i < 2 * kSy * S * 3 * kObN; i += NT) (&sm.ob[0][0][0][0])[i] = 0.f;
    for (int i = tid; i < 2 * kSy * 3 * kObT; i += NT) (&sm.obx[0][0][0][0])[i] = 0.f;
    // the pixels' channel values; absent pixels have no gradient, so they add nothing
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
        float2 l = make_float2(0.f, 0.f), gr = l, gc = l;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int y = Y + h * S;
            if (X < 0 || X >= wo || y < 0 || y >= ho) continue;
            const size_t o = ch * po + (size_t)y * wo + X;
            const float L = -lden[o], G = grad_rgb[o], GC = -G * rgb[o];
            if (h) { l.y = L; gr.y = G; gc.y = GC; }
            else { l.x = L; gr.x = G; gc.x = GC; }
        }
        sm.px[warp][ch][lane] = l;
        sm.px[warp][3 + ch][lane] = gr;
        sm.px[warp][6 + ch][lane] = gc;
    }
    RegionStage<SN, SD, NT, false> st(sm.st, burst, geo, g, kern, rhat_planes, blockIdx.x, blockIdx.y, tid);
    int rcx, rcy;
    float rfx = (float)stage::region_phase<SN, SD>(sx, rcx) * inv2Q, rfy = (float)stage::region_phase<SN, SD>(sy, rcy) * inv2Q;
    int ro = (v + 1 + rcy) * kTexP + u + 1 + rcx;
    int o0 = v * kTexP + u;
    const int m0 = v * kTexN + u, w0 = 2 * v * kRawP + u;
    const int wg = g.wh + kOff, hg = g.hh + kOff;
    const bool in0 = U0 + u >= -kOff && U0 + u < g.wh && V0 + v >= -kOff && V0 + v < g.hh;
    const bool in1 = U0 + u >= -kOff && U0 + u < g.wh && V0 + v + 1 >= -kOff && V0 + v + 1 < g.hh;
    int rp = (V0 + v + kOff) * wg + U0 + u + kOff;  // in the phase's plane
    stage::keep(ro); stage::keep(o0); stage::keep(rp);
    // who gathers: along x every thread, (y phase, entry, row, column) items; along y the last 128
    // threads (all where there are fewer), a texel or two each
    constexpr int kGy0 = NT >= 128 ? NT - 128 : 0, kGyL = NT >= 128 ? 1 : (kTexN * kTexN + NT - 1) / NT;
    constexpr int kGx = kSy * 3 * 8 * kTexN, kGxL = (kGx + NT - 1) / NT;
    int gidx[kGxL];  // source | destination << 16
#pragma unroll
    for (int k = 0; k < kGxL; ++k) {
        const int i = tid + k * NT, cc = i % kTexN, q = i / kTexN, row = q & 7, e = q >> 3;  // e = y phase x 3 + entry
        gidx[k] = ((e / 3) * S * 3 * kObN + (e % 3) * kObN + 2 + row * kTexP + cc + 2) | (e * kObT + (row + 3) * kTexP + cc) << 16;
        if (i >= kGx) gidx[k] = -1;
        stage::keep(gidx[k]);
    }
    int tex[kGyL];  // row | column << 8
#pragma unroll
    for (int k = 0; k < kGyL; ++k) {
        const int i = tid - kGy0 + k * NT, r = i / kTexN;
        tex[k] = i >= 0 && i < kTexN * kTexN ? r | (i - r * kTexN) << 8 : -1;

    }
    float pb[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const float2 neg1 = make_float2(-1.f, -1.f);

    // Three stages run side by side, a frame apart, with one barrier per step: the pixels of frame
    // `it`, the gather along x of frame it - 1, and along y (and the kernel shape) of frame it - 2.
    st.begin(0);
    for (int it = 0; it < g.n + 2; ++it) {
        const int b = it & 1;
        if (it >= 1 && it - 1 < g.n) {  // the texels' shape in frame it - 1, for the next step
            const typename RegionSmem<S>::Desc &d = st.desc(it - 1);
            const float4 *p = shape + (d.tex - kern);
#pragma unroll
            for (int k = 0; k < kGyL; ++k) {
                const int tr = tex[k] & 255, tc = tex[k] >> 8;
                if (tex[k] < 0) continue;
                const int o = d.cx == INT_MIN ? tr * g.wh + tc
                                              : clampi(d.cy + tr, 0, g.hh - 1) * g.wh + clampi(d.cx + tc, 0, g.wh - 1);
                stage::copy16(&sm.sh[b ^ 1][tr * kTexN + tc], p + o);
            }
        }
        if (it < g.n) {
            const int f = stage::frame_of_step(it, g.ref);
            st.template ahead<2>(it, 0);
            const typename RegionSmem<S>::Frame &fr = sm.st.fr[b];
            float2 rh = make_float2(1.f, 1.f);
            if (it > 0) {
                const float *R = fr.rh + ro;
                const float rfx1 = 1.f - rfx, rfy1 = 1.f - rfy;
                const float h0 = fmaf(rfx, R[1], rfx1 * R[0]), h1 = fmaf(rfx, R[kTexP + 1], rfx1 * R[kTexP]);
                const float h2 = fmaf(rfx, R[2 * kTexP + 1], rfx1 * R[2 * kTexP]);
                rh = make_float2(fmaf(rfy, h1, rfy1 * h0), fmaf(rfy, h2, rfy1 * h1));
            }
            const AxisTab &tx = sm.st.tab[it & (kRing - 1)][sx], &ty = sm.st.tab[it & (kRing - 1)][S + sy];
            const float4 qx = tx.q, qy = ty.q, fx = tx.fr, fy = ty.fr;
            const int kx = __float_as_int(qx.w), ky = __float_as_int(qy.w);
            const bool hix = (kx & 256) != 0, hiy = (ky & 256) != 0;
            const int o = o0 + (kx & 255) + (ky & 255) * kTexP, m = m0 + (kx & 255) + (ky & 255) * kTexN;
            // Omega at the pixels, its inverse, and its derivatives along the sampling position
            float2 Sxx, Syy, Sxy;             // Omega^-1
            float2 xa[2], xb[2], ya[2], yb[2];  // d{a, Myy}, d{-2 Mxy, Mxx} / d fraction along x, y, per pixel
            {
                float2 l[3], r[3], dl[3], dr[3];
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const float4 t0 = fr.om[m + j * kTexN], t1 = fr.om[m + j * kTexN + 1];
                    l[j] = fma2(hi2(fx), lo2(t1), mul2(lo2(fx), lo2(t0)));
                    r[j] = fma2(hi2(fx), hi2(t1), mul2(lo2(fx), hi2(t0)));
                    dl[j] = fma2(neg1, lo2(t0), lo2(t1));
                    dr[j] = fma2(neg1, hi2(t0), hi2(t1));
                }
                const float ch[3] = {fr.ch[o], fr.ch[o + kTexP], fr.ch[o + 2 * kTexP]};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float2 L = fma2(hi2(fy), l[h + 1], mul2(lo2(fy), l[h])), R = fma2(hi2(fy), r[h + 1], mul2(lo2(fy), r[h]));
                    xa[h] = fma2(hi2(fy), dl[h + 1], mul2(lo2(fy), dl[h]));
                    xb[h] = fma2(hi2(fy), dr[h + 1], mul2(lo2(fy), dr[h]));
                    ya[h] = fma2(neg1, l[h], l[h + 1]);
                    yb[h] = fma2(neg1, r[h], r[h + 1]);
                    const float u1 = fmaf(qy.z, ch[h + 1], qy.y * ch[h]);
                    const float u2 = fmaf(qx.x, fr.cd[o + h * kTexP],
                                          fmaf(qx.z, fr.cv[o + h * kTexP + 1], qx.y * fr.cv[o + h * kTexP]));
                    const float dM = fmaf(qx.x, u1, qy.x * u2);
                    const float s1 = L.x + L.y;
                    const float det = fmaf(L.x, s1 + R.y, dM);
                    const float r0 = fast_rcp(det), id = fmaf(fmaf(-det, r0, 1.f), r0, r0);
                    const float vx = s1 * id, vy = (L.x + R.y) * id, vxy = 0.5f * R.x * id;
                    if (h) { Sxx.y = vx; Syy.y = vy; Sxy.y = vxy; }
                    else { Sxx.x = vx; Syy.x = vy; Sxy.x = vxy; }
                }
            }
            const float4 dxa = tx.d01, dya = ty.d01;
            const float2 dx[3] = {lo2(dxa), hi2(dxa), lo2(tx.d2s0)}, dy[3] = {lo2(dya), hi2(dya), lo2(ty.d2s0)};
            // the channels of the window's sample classes: C centre, H (+-1, 0), V (0, +-1), K corners
            const int ox = hix ? 0 : 1, oy = hiy ? 0 : 1;
            const int cls[4] = {ox + oy, 1 - ox + oy, ox + 1 - oy, 2 - ox - oy};
            const float *W = fr.raw + (w0 + (kx & 255) + 2 * kRawP * (ky & 255) + (hiy ? kRawP : 0));
            const float *Wc[3] = {W + (hix ? kRawOdd : 0), W + (hix ? 1 : kRawOdd), W + (hix ? kRawOdd + 1 : 1)};
            bool xok[3] = {true, true, true}, yok[5] = {true, true, true, true, true};
            const bool border = (kx & 512) != 0;
            if (border) {
                const typename RegionSmem<S>::Desc &d = st.desc(it);
                const int ax = 2 * (d.cx + u + (kx & 255)) + (hix ? 1 : 0), ay = 2 * (d.cy + v + (ky & 255)) + (hiy ? 1 : 0);
#pragma unroll
                for (int i = 0; i < 3; ++i) xok[i] = (unsigned)(ax + i) < (unsigned)g.w;
#pragma unroll
                for (int j = 0; j < 5; ++j) yok[j] = (unsigned)(ay + j) < (unsigned)g.h;
            }
            const float2 nk = make_float2(-stage::kHalfLog2e, -stage::kHalfLog2e);
            float2 sPx = make_float2(0.f, 0.f), sPy = sPx, o00 = sPx, o01 = sPx, o11 = sPx, rhb = sPx;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int i = q == 2 ? 1 : 2 * q;  // the outer columns first: they share their two classes
                float2 nL[4], G[4], nGC[4];
#pragma unroll
                for (int k = i == 1 ? 0 : 1; k < 4; k += 2) {
                    nL[k] = sm.px[warp][cls[k]][lane];
                    G[k] = sm.px[warp][3 + cls[k]][lane];
                    nGC[k] = sm.px[warp][6 + cls[k]][lane];
                }
                const float2 pxc = mul2(Sxx, dx[i]), pyc = mul2(Sxy, dx[i]), dxk = mul2(nk, dx[i]);
                float val[5];
#pragma unroll
                for (int j = 0; j < 5; ++j) val[j] = Wc[i][j * kRawP];
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const int k = i == 1 ? (j == 1 ? 0 : 2) : (j == 1 ? 1 : 3);
                    const float2 Px = fma2(Sxy, dy[j], pxc), Py = fma2(Syy, dy[j], pyc);  // Omega^-1 d
                    const float2 dyk = mul2(nk, dy[j]);
                    const float2 t = fma2(dxk, Px, fma2(dyk, Py, nL[k]));  // log2 of the weight over its channel's sum
                    float2 w = make_float2(fast_exp2(t.x), fast_exp2(t.y));
                    if (border) {
                        if (!(xok[i] && yok[j])) w.x = 0.f;
                        if (!(xok[i] && yok[j + 2])) w.y = 0.f;
                    }
                    const float2 gv = fma2(G[k], make_float2(val[j], val[j + 2]), nGC[k]);  // dL/d(w Rhat)
                    rhb = fma2(gv, w, rhb);
                    const float2 e = mul2(gv, mul2(w, rh));  // times w Rhat, which is at most 1
                    const float2 t1 = mul2(e, Px), t2 = mul2(e, Py);
                    sPx = add2(sPx, t1);
                    sPy = add2(sPy, t2);
                    o00 = fma2(t1, Px, o00);
                    o01 = fma2(t1, Py, o01);
                    o11 = fma2(t2, Py, o11);
                }
            }
            // Omega-bar = sum e P P^T / 2 (o01 doubled: the entry stands for both); the offsets give
            // dL/dv = sum e P.  A frame rejected at a pixel is not in its channels' sums, so its w has
            // no bound: it is left out here, where 0 times it (or times its product with P) may be no
            // number.
            const float2 half = make_float2(0.5f, 0.5f);
            o00 = mul2(o00, half);
            o11 = mul2(o11, half);
            if (!(rh.x > 0.f)) o00.x = o01.x = o11.x = sPx.x = sPy.x = 0.f;
            if (!(rh.y > 0.f)) o00.y = o01.y = o11.y = sPx.y = sPy.y = 0.f;
            float *ob = &sm.ob[b][warp][0][2 + v * kTexP + u + 2];
            ob[0] = o00.x; ob[kTexP] = o00.y;
            ob[kObN] = o01.x; ob[kObN + kTexP] = o01.y;
            ob[2 * kObN] = o11.x; ob[2 * kObN + kTexP] = o11.y;
            if (it > 0) {
                const float2 part = make_float2(kPart, kPart);
                float2 vx = mul2(sPx, part), vy = mul2(sPy, part);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    // through Omega's sampling position (half a texel per raw px)
                    const float A0 = h ? o00.y : o00.x, A1 = h ? o01.y : o01.x, A2 = h ? o11.y : o11.x;
                    const float tr2 = A0 + A2, mA1 = -0.5f * A1;
                    const float px = fmaf(tr2, xa[h].x, fmaf(A2, xa[h].y, fmaf(mA1, xb[h].x, A0 * xb[h].y)));
                    const float py = fmaf(tr2, ya[h].x, fmaf(A2, ya[h].y, fmaf(mA1, yb[h].x, A0 * yb[h].y)));
                    if (h) { vx.y = fmaf(0.5f * kPart, px, vx.y); vy.y = fmaf(0.5f * kPart, py, vy.y); }
                    else { vx.x = fmaf(0.5f * kPart, px, vx.x); vy.x = fmaf(0.5f * kPart, py, vy.x); }
                }
                // the warp's sums: lanes 0-15 take x, 16-31 y; every addition's rounding error is
                // carried along (two-sum), from the lane's two pixels on
                const bool lo = lane < 16;
                float a = lo ? vx.x : vy.x, ae = 0.f, o2 = lo ? vy.x : vx.x, oe = 0.f;
                two_sum(a, ae, lo ? vx.y : vy.y, 0.f);
                two_sum(o2, oe, lo ? vy.y : vx.y, 0.f);
                two_sum(a, ae, __shfl_xor_sync(0xffffffffu, o2, 16), __shfl_xor_sync(0xffffffffu, oe, 16));
#pragma unroll
                for (int q = 8; q > 0; q >>= 1)
                    two_sum(a, ae, __shfl_xor_sync(0xffffffffu, a, q), __shfl_xor_sync(0xffffffffu, ae, q));
                if ((lane & 15) == 0)
                    vbar_region[(((((size_t)f * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * gridDim.z + blockIdx.z) * NW + warp) * 2 + (lane >> 4)] =
                        make_float2(a, error_of(a, ae));
                float *plane = rhbar_phase + ((size_t)f * (S * S) + (size_t)(sy * S + sx)) * ((size_t)hg * wg);
                if (in0) plane[rp] = rhb.x;
                if (in1) plane[rp + wg] = rhb.y;
            }
        }
        // dL/dOmega onto texel columns ...
        if (it >= 1 && it - 1 < g.n) {
            const AxisTab *tx = sm.st.tab[(it - 1) & (kRing - 1)];
#pragma unroll
            for (int k = 0; k < kGxL; ++k) {
                if (gidx[k] < 0) continue;
                const float *src = &sm.ob[b ^ 1][0][0][0] + (gidx[k] & 0xffff);
                float acc = 0.f;
#pragma unroll
                for (int p = 0; p < S; ++p) {
                    const float *q = src + p * 3 * kObN - (__float_as_int(tx[p].q.w) & 255);
                    acc = fmaf(tx[p].fr.x, q[0], fmaf(tx[p].fr.z, q[-1], acc));
                }
                (&sm.obx[b ^ 1][0][0][0])[gidx[k] >> 16] = acc;
            }
        }
        // ... and rows, and through the texel's kernel shape into the parameters
        if (it >= 2) {
            const AxisTab *ty = sm.st.tab[(it - 2) & (kRing - 1)] + S + blockIdx.z * kSy;
#pragma unroll
            for (int i = 0; i < kGyL; ++i) {
                if (tex[i] < 0) continue;
                const int at = ((tex[i] & 255) + 3) * kTexP + (tex[i] >> 8);
                float A[3] = {0.f, 0.f, 0.f};
#pragma unroll
                for (int p = 0; p < kSy; ++p) {
                    const float *q = &sm.obx[b][p][0][0] + at - (__float_as_int(ty[p].q.w) & 255) * kTexP;
                    const float w1 = ty[p].fr.x, w2 = ty[p].fr.z;
#pragma unroll
                    for (int k = 0; k < 3; ++k) A[k] = fmaf(w1, q[k * kObT], fmaf(w2, q[k * kObT - kTexP], A[k]));
                }
                const float4 t = sm.sh[b][(tex[i] & 255) * kTexN + (tex[i] >> 8)];
                const float oE1 = fmaf(A[0], 0.5f * (1.f + t.z), fmaf(A[1], 0.5f * t.w, A[2] * (0.5f * (1.f - t.z))));
                kernel_grad_acc(t, c, kc, oE1, (A[0] + A[2]) - oE1, pb);
            }
        }
        if (it + 1 < g.n) st.advance(it);
        else {
            stage::copy_wait();
            __syncthreads();
        }
    }
    // block sums of the six kernel-parameter gradients, in a fixed order
    float pe[6];
    warp_sums_comp<6>(pb, pe);
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            sm.red[warp][2 * q] = (double)pb[q];
            sm.red[warp][2 * q + 1] = (double)pe[q];
        }
    __syncthreads();
    if (tid < 6) {
        double acc = 0.0;
        for (int w = 0; w < NW; ++w) acc += sm.red[w][2 * tid] + sm.red[w][2 * tid + 1];
        const size_t bid = ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        partials[bid * 6 + tid] = acc;
    }
}

// ---------------------------------------------------------------------------------------
// Rhat-bar onto base texels (the transpose of the forward's bilinear sampling, by phases), then
// through the 5x5 argmin into R's parameters and the motion: one block of 32 x 16 texels, with the
// 2-texel halo whose windows may have picked its texels.  The Rhat-bar of a texel never leaves
// shared memory.
// ---------------------------------------------------------------------------------------
constexpr int kRpW = 32, kRpH = 16, kRpHaloW = kRpW + 4, kRpHaloH = kRpH + 4;

// the taps along one axis of texel t from output pixels of phase s: grid indices (texel of the
// pixel + kOff) and weights (a clamped cell has both its weights on the border texel)
template <int SN, int SD>
__device__ __forceinline__ void rhat_phase_taps(int t, int nt, int s, int (&idx)[2], float (&w)[2]) {
    constexpr int kOff = RegionScale<SN, SD>::kOff;
    constexpr float inv2Q = 0.25f / (float)SN;
    int rc;
    const float f = (float)stage::region_phase<SN, SD>(s, rc) * inv2Q;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int q = t - rc - k, cell = q + rc;
        const bool ok = q >= -kOff && q < nt;
        idx[k] = ok ? q + kOff : 0;
        w[k] = ok ? (clampi(cell, 0, nt - 1) == t ? 1.f - f : 0.f) + (clampi(cell + 1, 0, nt - 1) == t ? f : 0.f) : 0.f;
    }
}

template <int SN, int SD>
__global__ void __launch_bounds__(kRpW *kRpH) k_rpath_region(const float *__restrict__ rhbar_phase,
                                                             const unsigned char *__restrict__ flags,
                                                             const float4 *__restrict__ rb, Geom g,
                                                             float4 *__restrict__ vbar_block,
                                                             double *__restrict__ partials) {
    constexpr int S = RegionScale<SN, SD>::S, kOff = RegionScale<SN, SD>::kOff;
    __shared__ float s_x[S][kRpHaloH + 1][kRpHaloW];
    __shared__ float2 s_rh[kRpHaloH][kRpHaloW];  // Rhat-bar, and the code of the offset its window picked
    __shared__ double s_red[kRpH][4];
    __shared__ float4 s_vb[kRpH][4];  // {x, its error, y, its error}
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, f = blockIdx.z;
    const int u0 = blockIdx.x * kRpW, v0 = blockIdx.y * kRpH;
    const size_t hw = (size_t)g.hh * g.wh;
    const size_t bid = ((size_t)f * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    if (f == g.ref) {  // the whole block
        if (threadIdx.x < 2) partials[bid * 2 + threadIdx.x] = 0.0;
        return;
    }
    const int wg = g.wh + kOff;
    const size_t plane = (size_t)(g.hh + kOff) * wg;
    const float *Pf = rhbar_phase + (size_t)f * (S * S) * plane;
    // along x, for each y phase: the pixel rows that the taps of texel rows v0 - 2 .. v0 + kRpH + 1
    // touch.  Away from the border a phase's two taps and weights are constants.  A pixel of weight 0
    // is left out, so that one without a finite gradient reaches no texel that it does not sample.
    constexpr int kRows = kRpHaloH + 1;
    constexpr float inv2Q = 0.25f / (float)SN;
    for (int i = threadIdx.x; i < S * kRows * kRpHaloW; i += kRpW * kRpH) {
        const int q = i / kRpHaloW, cc = i - q * kRpHaloW, sy = q / kRows, r = q - sy * kRows;
        int rcy;
        stage::region_phase<SN, SD>(sy, rcy);
        const int uu = u0 - 2 + cc, row = v0 - 3 - rcy + r;
        float acc = 0.f;
        if (uu >= 0 && uu < g.wh && row >= -kOff && row < g.hh) {
            const float *p = Pf + (size_t)(sy * S) * plane + (size_t)(row + kOff) * wg;
            if (uu >= 1 && uu + 1 < g.wh) {
#pragma unroll
                for (int sx = 0; sx < S; ++sx) {
                    int rc;
                    const float w = (float)stage::region_phase<SN, SD>(sx, rc) * inv2Q;
                    const float *ps = p + (size_t)sx * plane + (uu - rc + kOff);
                    if (w != 0.f) acc = fmaf(w, __ldg(ps - 1), acc);
                    acc = fmaf(1.f - w, __ldg(ps), acc);
                }
            } else {
#pragma unroll
                for (int sx = 0; sx < S; ++sx) {
                    int ix[2];
                    float wx[2];
                    rhat_phase_taps<SN, SD>(uu, g.wh, sx, ix, wx);
                    const float *ps = p + (size_t)sx * plane;
                    if (wx[1] != 0.f) acc = fmaf(wx[1], __ldg(ps + ix[1]), acc);
                    if (wx[0] != 0.f) acc = fmaf(wx[0], __ldg(ps + ix[0]), acc);
                }
            }
        }
        s_x[sy][r][cc] = acc;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kRpHaloW * kRpHaloH; i += kRpW * kRpH) {
        const int r = i / kRpHaloW, cc = i - r * kRpHaloW, uu = u0 - 2 + cc, vv = v0 - 2 + r;
        float acc = 0.f;
        int fl = 31;  // no texel's window
        if (uu >= 0 && uu < g.wh && vv >= 0 && vv < g.hh) {
            fl = flags[(size_t)f * hw + (size_t)vv * g.wh + uu];
            // pixel rows vv - rcy (r + 1 of s_x) and vv - rcy - 1 (r)
#pragma unroll
            for (int sy = 0; sy < S; ++sy) {
                int iy[2];
                float wy[2];
                rhat_phase_taps<SN, SD>(vv, g.hh, sy, iy, wy);
                if (wy[1] != 0.f) acc = fmaf(wy[1], s_x[sy][r][cc], acc);
                if (wy[0] != 0.f) acc = fmaf(wy[0], s_x[sy][r + 1][cc], acc);
            }
        }
        s_rh[r][cc] = make_float2(acc, __int_as_float(fl));
    }
    __syncthreads();
    const int u = u0 + tx, v = v0 + ty;
    float pv[2] = {0.f, 0.f}, pe[2], vb[2] = {0.f, 0.f}, ve[2];
    if (u < g.wh && v < g.hh) {
        // R-bar(u, v): the windows centred at (u + i, v + j) that picked offset (-i, -j)
        float rbar = 0.f;
#pragma unroll
        for (int j = -2; j <= 2; ++j)
#pragma unroll
            for (int i = -2; i <= 2; ++i)
            {
                const float2 q = s_rh[ty + 2 + j][tx + 2 + i];
                if ((__float_as_int(q.y) & 31) == (2 - j) * 5 + (2 - i)) rbar += q.x;
            }
        if (__float_as_int(s_rh[ty + 2][tx + 2].y) & 0x80) {  // R unclamped
            const float4 d = rb[(size_t)f * hw + (size_t)v * g.wh + u];
            vb[0] = kPart * (rbar * d.y);
            vb[1] = kPart * (rbar * d.z);
            pv[0] = rbar * d.w;
            pv[1] = -rbar;
        }
    }
    // 8 x 8-texel sums of the motion contributions
    warp_sums_comp<2, 8>(vb, ve);
    if ((tx & 7) == 0) s_vb[ty][tx >> 3] = make_float4(vb[0], ve[0], vb[1], ve[1]);
    warp_sums_comp<2>(pv, pe);
    if (tx == 0) {
        s_red[ty][0] = (double)pv[0]; s_red[ty][1] = (double)pe[0];
        s_red[ty][2] = (double)pv[1]; s_red[ty][3] = (double)pe[1];
    }
    __syncthreads();
    if (threadIdx.x < 4 * kRpH) {  // a lane's row of a block: four blocks' rows in a warp
        const int k = threadIdx.x & 3, r = threadIdx.x >> 2;
        const float4 q = s_vb[r][k];
        float x = q.x, xe = q.y, y = q.z, ye = q.w;
#pragma unroll
        for (int o = 4; o < 32; o *= 2) {
            two_sum(x, xe, __shfl_xor_sync(0xffffffffu, x, o), __shfl_xor_sync(0xffffffffu, xe, o));
            two_sum(y, ye, __shfl_xor_sync(0xffffffffu, y, o), __shfl_xor_sync(0xffffffffu, ye, o));
        }
        const int bx = blockIdx.x * 4 + k, by = blockIdx.y * (kRpH / 8) + (r >> 3);
        const int nbx = div_up(g.wh, 8), nby = div_up(g.hh, 8);
        if ((r & 7) == 0 && bx < nbx && by < nby)
            vbar_block[((size_t)f * nby + by) * nbx + bx] = make_float4(x, error_of(x, xe), y, error_of(y, ye));
    } else if (threadIdx.x < 4 * kRpH + 2) {
        const int q = threadIdx.x - 4 * kRpH;
        double acc = 0.0;
        for (int r = 0; r < kRpH; ++r) acc += s_red[r][2 * q] + s_red[r][2 * q + 1];
        partials[bid * 2 + q] = acc;
    }
}

// Every tile's motion gradient: its regions' and its 8 x 8-texel blocks' sums, in a fixed order, in
// FP64; their rounding errors, 2^-24 of them and less, in FP32 beside it.  Eight lanes per tile, so
// that a tile's loads (up to 16 parts of each region) are in flight together: latency and the FP64
// additions are all of it.  1 MP x 8 at 3/2: 16 us (20 with the errors in FP64 too); the
// 256 x 320 x 4 crop at 2x: 7 us (23 with one lane per tile).
constexpr int kTileLanes = 8;
__global__ void __launch_bounds__(128) k_motion_region(const float2 *__restrict__ vbar_region, const float4 *__restrict__ vbar_block,
                                                       Geom g, int off, int parts, float2 *__restrict__ grad_motion) {
    const int t = (blockIdx.x * 128 + threadIdx.x) / kTileLanes, l = threadIdx.x % kTileLanes;
    const int ntl = g.ty * g.tx, f = t / ntl, r = t - f * ntl, ty = r / g.tx, tx = r - ty * g.tx;
    double x = 0.0, y = 0.0;
    float xe = 0.f, ye = 0.f;
    if (t < g.n * ntl && f != g.ref) {
        const int nb = g.tile / 16, nbx = div_up(g.wh, 8), nby = div_up(g.hh, 8);
        const int x0 = tx * nb, y0 = ty * nb, bw = min(x0 + nb, nbx) - x0, bh = min(y0 + nb, nby) - y0;
        for (int k = l; k < bw * bh; k += kTileLanes) {
            const int by = k / bw, bx = k - by * bw;
            const float4 q = __ldg(vbar_block + ((size_t)f * nby + y0 + by) * nbx + x0 + bx);
            x += (double)q.x;
            y += (double)q.z;
            xe += q.y;
            ye += q.w;
        }
        // regions are the same 8 x 8 texels, after `off` leading ones that belong to the first tiles
        const int nrx = nbx + off, nry = nby + off;
        const int rx0 = tx == 0 ? 0 : x0 + off, ry0 = ty == 0 ? 0 : y0 + off, rw = x0 + bw + off - rx0, rh = y0 + bh + off - ry0;
        for (int k = l; k < rw * rh * parts; k += kTileLanes) {  // a warp's sums, each with its rounding error
            const int q0 = k / parts, by = q0 / rw, bx = q0 - by * rw;
            const float4 q = __ldg(reinterpret_cast<const float4 *>(vbar_region) +
                                   (((size_t)f * nry + ry0 + by) * nrx + rx0 + bx) * parts + (k - q0 * parts));
            x += (double)q.x;
            y += (double)q.z;
            xe += q.y;
            ye += q.w;
        }
    }
    x += (double)xe;
    y += (double)ye;
#pragma unroll
    for (int o = kTileLanes / 2; o > 0; o >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    constexpr double kWhole = 1.0 / kPart;
    if (l == 0 && t < g.n * ntl) grad_motion[t] = make_float2((float)(kWhole * x), (float)(kWhole * y));
}

template <int SN, int SD>
cudaError_t launch_main(const uint16_t *burst, const Geom &g, const MergeConsts &c, const MergePlanes &P,
                        const BwdPlanes &B, int ho, int wo, const float *rgb, const float *lden, const float *grad_rgb,
                        cudaStream_t s) {
    constexpr int S = RegionScale<SN, SD>::S, kSy = AdjointShape<SN, SD>::kSy;
    constexpr size_t bytes = sizeof(AdjointSmem<S, kSy>);
    const cudaError_t e = cudaFuncSetAttribute(k_adjoint_region<SN, SD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    k_adjoint_region<SN, SD><<<dim3(stage::region_count<SN, SD>(g.w), stage::region_count<SN, SD>(g.h), S / kSy),
                               32 * kSy * S, bytes, s>>>(burst, P.geo, g, c, kconsts_of(c), P.kern, B.shape, P.rhat, ho, wo, rgb, lden,
                                                         grad_rgb, B.rhbar_phase, B.vbar_region, B.part6);
    return cudaGetLastError();
}

template <int SN, int SD>
BwdRegionSizes sizes(const Geom &g) {
    constexpr int S = RegionScale<SN, SD>::S, kOff = RegionScale<SN, SD>::kOff;
    BwdRegionSizes z;
    const size_t regions = (size_t)stage::region_count<SN, SD>(g.w) * stage::region_count<SN, SD>(g.h);
    constexpr int parts = S / AdjointShape<SN, SD>::kSy;
    z.rhbar = (size_t)g.n * S * S * (size_t)(g.hh + kOff) * (g.wh + kOff);
    z.vregion = (size_t)g.n * regions * S * S * 2;
    z.vblock = (size_t)g.n * div_up(g.wh, 8) * div_up(g.hh, 8);
    z.bwd_blocks = (int)(regions * parts);
    z.rp_blocks = div_up(g.wh, kRpW) * div_up(g.hh, kRpH) * g.n;
    return z;
}

template <int SN, int SD>
cudaError_t launch_finish(const Geom &g, const BwdPlanes &B, float *grad_motion, cudaStream_t s) {
    constexpr int S = RegionScale<SN, SD>::S, kOff = RegionScale<SN, SD>::kOff;
    k_rpath_region<SN, SD><<<dim3(div_up(g.wh, kRpW), div_up(g.hh, kRpH), g.n), kRpW * kRpH, 0, s>>>(
        B.rhbar_phase, B.flags, B.rb, g, B.vbar_block, B.part2);
    k_motion_region<<<div_up(g.n * g.ty * g.tx * kTileLanes, 128), 128, 0, s>>>(B.vbar_region, B.vbar_block, g, kOff, S * S,
                                                                 reinterpret_cast<float2 *>(grad_motion));
    return cudaGetLastError();
}

}  // namespace

bool bwd_region(const Geom &g, int snum, int sden) { return stage::region_kind(g.tile, snum, sden) != 0; }

BwdRegionSizes bwd_region_sizes(const Geom &g, int snum, int sden) {
    switch (stage::region_kind(g.tile, snum, sden)) {
        case 1: return sizes<1, 1>(g);
        case 2: return sizes<3, 2>(g);
        default: return sizes<2, 1>(g);
    }
}

cudaError_t launch_bwd_region_main(const uint16_t *burst, const float *motion, const Geom &g, const MergeConsts &c,
                                   const MergePlanes &P, const BwdPlanes &B, int snum, int sden, const float *rgb,
                                   const float *lden, const float *grad_rgb, cudaStream_t s) {
    const int ho = (int)(((long long)g.h * snum) / sden), wo = (int)(((long long)g.w * snum) / sden);
    // the table depends on the scale, so it is written here also where the planes are prepared
    const cudaError_t e = launch_geo(motion, g, P, snum, sden, s);
    if (e != cudaSuccess) return e;
    switch (stage::region_kind(g.tile, snum, sden)) {
        case 1: return launch_main<1, 1>(burst, g, c, P, B, ho, wo, rgb, lden, grad_rgb, s);
        case 2: return launch_main<3, 2>(burst, g, c, P, B, ho, wo, rgb, lden, grad_rgb, s);
        default: return launch_main<2, 1>(burst, g, c, P, B, ho, wo, rgb, lden, grad_rgb, s);
    }
}

cudaError_t launch_bwd_region_finish(const Geom &g, const BwdPlanes &B, int snum, int sden, float *grad_motion,
                                     cudaStream_t s) {
    switch (stage::region_kind(g.tile, snum, sden)) {
        case 1: return launch_finish<1, 1>(g, B, grad_motion, s);
        case 2: return launch_finish<3, 2>(g, B, grad_motion, s);
        default: return launch_finish<2, 1>(g, B, grad_motion, s);
    }
}

}  // namespace hmfsr
