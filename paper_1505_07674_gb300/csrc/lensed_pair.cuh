// The ray loop of the FP32 first pass (a2-a5) for two pixels of one thread.
//
// The path is bound by instruction issue and the FMA pipe, not by memory, so
// the loop is laid out to issue as few instructions per ray as it can while
// every ray keeps the bits of the one-pixel form (sie_row_v, light_row_v):
//   - a thread owns two pixels and every value is a pair (one per pixel), so
//     all arithmetic that has a packed form uses it, whatever the rule's node
//     count (rays paired inside a row leave one of five alone);
//   - C <= 4 rays of a node row are traced together component by component;
//     their constants are read once per 2 C rays, from shared memory, in the
//     form the loop uses them (negations included, components sorted into
//     lenses and lights by stage_pair);
//   - psi is clamped from below once, which covers the divisions after it;
//   - both forms of atanh are evaluated for every ray and one is selected:
//     5 packed operations more than branching, but no branch splits the C
//     chains, which lets them overlap in 80 registers (6 warps per
//     scheduler).
// Measured on the 200x200 workload (5 x 5 rule, 512 points): 87 warp
// instructions per 32 rays, 44 of them packed, first pass 705 us; 941 us with
// one pixel per thread.  A packed operation takes two issue slots: 131 of the
// 131 scheduler cycles per 32 rays.  7 x 7 rays, eight components: 91 % of the
// cycles; the rest waits for instructions (0.81 such stalls per issue, 0.17
// with the 5 x 5 rule): its code holds a chunk of 4 and one of 3 rays.
#pragma once

#include "lensed_internal.cuh"
#include "lensed_sie_trig.cuh"

namespace lensed {

// MIXED_FF re-traces rays with (R / r)^2 below this.  Measured against the
// oracle (225 prior points of the 200x200 workload, 256 of the 64x64 one),
// R < r/2 leaves the largest log-likelihood errors as low as R < r does
// (7.2e-4 and 4.7e-4 against 9.3e-4 and 3.7e-4: the worst points are set by
// other float terms) at a quarter of the re-traced rays; below it they grow
// (R < 0.32 r: 1.1e-3, R < 0.2 r: 3.1e-3 on the 200x200 sample).
constexpr float kCuspRho2 = 0.25f;

// Staged constants of one component: the packed FP32 block (k_prologue_comp)
// with -x0, -y0 in slots 0 and 1, and two more values behind it
// (lights and SIE: -sin PA and its residual; shear: -gamma_1).
constexpr int kPairNC = 28;
constexpr int kPairNSn = 24, kPairNSnL = 25;

constexpr int kPairW = 8;  // row stride of the staged 2-D weights (16-byte rows)

struct PairSmem {
    float cf[LENSED_MAX_COMPONENTS * kPairNC];
    // the lens components (offset into cf << 8 | type), the lights evaluated
    // at the image position, and the sources, each in component order
    int lens[LENSED_MAX_COMPONENTS], light[LENSED_MAX_COMPONENTS];
    int n_lens, n_fore, n_light;  // light: n_fore foreground ones, then the sources
    float u[LENSED_MAX_RULE_ORDER];
    float w[LENSED_MAX_RULE_ORDER * LENSED_MAX_RULE_ORDER];
};

// Stage one (system, point): every thread of the CTA takes part; a barrier
// follows.  wstride: floats per row of w (nn, or kPairW for a rule of at
// most 8 nodes per row).
__device__ __forceinline__ void stage_pair(PairSmem &sm, const SysDev &S,
                                           const int *__restrict__ comp_type,
                                           const int *__restrict__ comp_plane,
                                           const float *__restrict__ cf, size_t cbase,
                                           const NodeTables &nodes, int wstride)
{
    const int ncomp = S.ncomp, nn = S.nn;
    for (int k = threadIdx.x; k < ncomp * kPairNC; k += blockDim.x) {
        const int c = k / kPairNC, e = k - c * kPairNC;
        const float *src = cf + cbase + (size_t)c * kNC;
        const int t = comp_type[S.comp_off + c];
        float v = 0.f;
        if (e < 2) v = -src[e];
        else if (e < kNC) v = src[e];
        else if (e == kPairNSn) v = t == LENSED_SHEAR ? -src[2] : -src[3];
        else if (e == kPairNSnL) v = -src[5];
        sm.cf[k] = v;
    }
    if (threadIdx.x < 32u) {
        // one lane per component (at most 16), ranked within its list
        const int c = (int)threadIdx.x;
        const int pl = c < ncomp ? comp_plane[S.comp_off + c] : -1;
        const unsigned below = (1u << c) - 1u;
        const unsigned ml = __ballot_sync(0xffffffffu, pl == LENSED_PLANE_LENS);
        const unsigned mf = __ballot_sync(0xffffffffu, pl == LENSED_PLANE_FOREGROUND);
        const unsigned ms = __ballot_sync(0xffffffffu, pl == LENSED_PLANE_SOURCE);
        const int off = c * kPairNC;
        if (pl == LENSED_PLANE_LENS)
            sm.lens[__popc(ml & below)] = off << 8 | comp_type[S.comp_off + c];
        if (pl == LENSED_PLANE_FOREGROUND) sm.light[__popc(mf & below)] = off;
        if (pl == LENSED_PLANE_SOURCE) sm.light[__popc(mf) + __popc(ms & below)] = off;
        if (c == 0) {
            sm.n_lens = __popc(ml);
            sm.n_fore = __popc(mf);
            sm.n_light = __popc(mf) + __popc(ms);
        }
    }
    for (int k = threadIdx.x; k < nn; k += blockDim.x) sm.u[k] = nodes.u[S.node_off + k];
    for (int k = threadIdx.x; k < nn * nn; k += blockDim.x) {
        const int r = k / nn;
        sm.w[r * wstride + (k - r * nn)] = nodes.w[S.w2_off + k];
    }
}

__device__ __forceinline__ float2 sp(float s) { return make_float2(s, s); }

__device__ __forceinline__ float pair_rsqrt(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float pair_ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// NaN-propagating maximum
__device__ __forceinline__ float max_nan(float a, float b)
{
    float y;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
    return y;
}
// smallest of three in one instruction (sm_100 family)
__device__ __forceinline__ float min3(float a, float b, float c)
{
    float y;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
    return y;
}

// smallest normal float: below it the FP32 forms flush to zero
constexpr float kTiny = 1.17549435e-38f;

// atan(n / d), d > 0 (atan_ratio of lensed_sie_trig.cuh without its guard
// against d = 0)
__device__ __forceinline__ float2 pair_atan(float2 n, float2 d)
{
    const float2 lo = make_float2(fminf(fabsf(n.x), d.x), fminf(fabsf(n.y), d.y));
    const float2 rh = make_float2(trig_rcp(fmaxf(fabsf(n.x), d.x)), trig_rcp(fmaxf(fabsf(n.y), d.y)));
    const float2 t = vmul(lo, rh);
    const float2 u = vmul(t, t);
    const float2 r = vfma(vmul(t, u), minimax_atan_q(u), t);
    const float2 rc = vadd(vsub(sp(kHalfPiHi), r), sp(kHalfPiLo));
    return make_float2(copysignf(fabsf(n.x) > d.x ? rc.x : r.x, n.x),
                       copysignf(fabsf(n.y) > d.y ? rc.y : r.y, n.y));
}

// atanh(n / d), |n| < d: the polynomial up to |n / d| = 1/2, the logarithm
// beyond (atanh_ratio of lensed_sie_trig.cuh, both forms evaluated)
__device__ __forceinline__ float2 pair_atanh(float2 n, float2 d)
{
    const float2 z = vmul(n, make_float2(trig_rcp(d.x), trig_rcp(d.y)));
    const float2 m = vsub(d, n);
    const float2 q = vmul(vadd(d, n), make_float2(trig_rcp(m.x), trig_rcp(m.y)));
    const float2 L = make_float2(trig_lg2(q.x), trig_lg2(q.y));
    const float2 lg = vfma(sp(kHalfLn2Hi), L, vmul(sp(kHalfLn2Lo), L));
    const float2 u = vmul(z, z);
    const float2 P = vfma(vmul(z, u), minimax_atanh_q(u), z);
    return make_float2(u.x <= 0.25f ? P.x : lg.x, u.y <= 0.25f ? P.y : lg.y);
}

// Light at frame coordinates (u, v) of C ray pairs; R2: (R / r)^2.
struct LightP {
    float qr, iqr, qrl, iqrl, p2, B, Bl, A, Al, kind;
};
__device__ __forceinline__ LightP load_light_tail(const float *c)
{
    const float4 b = reinterpret_cast<const float4 *>(c)[1];
    const float4 d = reinterpret_cast<const float4 *>(c)[2];
    const float4 f = reinterpret_cast<const float4 *>(c)[3];
    return {b.z, b.w, d.x, d.y, d.z, d.w, f.x, f.y, f.z, f.w};
}
__device__ __forceinline__ float2 pair_light(const LightP &k, float2 u, float2 v, float2 &rho2)
{
    const float2 uu = vmul(u, u), vv = vmul(v, v);
    rho2 = vfma(sp(k.qr), uu, vfma(sp(k.iqr), vv, vfma(sp(k.qrl), uu, vmul(sp(k.iqrl), vv))));
    float2 f = rho2;
    if (k.kind != (float)kKindGauss) {
        f = vmul(sp(k.p2), make_float2(trig_lg2(rho2.x), trig_lg2(rho2.y)));
        f = make_float2(pair_ex2(f.x), pair_ex2(f.y));
    }
    const float2 t = vfma(sp(k.B), f, vmul(sp(k.Bl), f));
    const float2 g = make_float2(pair_ex2(-t.x), pair_ex2(-t.y));
    return vfma(sp(k.A), g, vmul(sp(k.Al), g));
}

// The deflection of one SIE for C rays of node row y of both pixels: set
// (FIRST) or added to (ax, ay).  ODD: the chunk's last ray is the last of a
// row with an odd number of nodes, whose psi is rounded before psi + s and
// psi + q^2 s are formed, as the one-pixel form's ray without a partner is
// (sie_row_v): the second pass and the in-block form give the same bits.
template <int C, bool FIRST, bool ODD>
__device__ __forceinline__ void pair_sie(const float *c, float2 y, float2 xc, const float (&u0)[C],
                                         float2 (&ax)[C], float2 (&ay)[C])
{
    const float4 a = reinterpret_cast<const float4 *>(c)[0];  // -x0 -y0 cs sn
    const float4 b = reinterpret_cast<const float4 *>(c)[1];  // cs_lo sn_lo q2 q2_lo
    const float4 d = reinterpret_cast<const float4 *>(c)[2];  // s2 s q2s e
    const float4 f = reinterpret_cast<const float4 *>(c)[3];  // e_lo pref pref_lo series
    const float2 g = reinterpret_cast<const float2 *>(c)[kPairNSn / 2];  // -sn -sn_lo
    const float2 dy = vadd(y, sp(a.y));
    const float2 rdu = vfma(dy, sp(a.w), vmul(dy, sp(b.y)));
    const float2 rdv = vfma(dy, sp(a.z), vmul(dy, sp(b.x)));
    float2 A1[C], A2[C];
#pragma unroll
    for (int k = 0; k < C; ++k) {
        const float2 dx = vadd(vadd(xc, sp(u0[k])), sp(a.x));
        const float2 u = vfma(dx, sp(a.z), vfma(dx, sp(b.x), rdu));
        const float2 v = vfma(dx, sp(g.x), vfma(dx, sp(g.y), rdv));
        const float2 w = vfma(u, u, sp(d.x));
        float2 p = vfma(sp(b.z), w, vfma(sp(b.w), w, vmul(v, v)));
        // psi^2 from the smallest normal float on: psi and both denominators
        // are then positive also at the very centre of a coreless SIE, where
        // u = v = 0 leaves no deflection
        p = make_float2(max_nan(p.x, kTiny), max_nan(p.y, kTiny));
        const float2 rs = make_float2(pair_rsqrt(p.x), pair_rsqrt(p.y));
        float2 du = vfma(p, rs, sp(d.y)), dv = vfma(p, rs, sp(d.z));
        if (ODD && k == C - 1) {
            const float px = __fmul_rn(p.x, rs.x), py = __fmul_rn(p.y, rs.y);
            du = make_float2(__fadd_rn(px, d.y), __fadd_rn(py, d.y));
            dv = make_float2(__fadd_rn(px, d.z), __fadd_rn(py, d.z));
        }
        if (f.w != 0.f) {
            // q -> 1: the series of sie_row_v, argument by argument
            const float e2 = c[16], e4 = __fmul_rn(e2, e2);
            A1[k] = vmap(u, du, [=](float uu, float dd) {
                const float z = __fdividef(uu, dd), z2 = __fmul_rn(z, z);
                return __fmul_rn(z, __fadd_rn(__fsub_rn(1.f, __fmul_rn(__fmul_rn(e2, z2), 1.f / 3.f)),
                                              __fmul_rn(__fmul_rn(__fmul_rn(e4, z2), z2), 0.2f)));
            });
            A2[k] = vmap(v, dv, [=](float vv, float dd) {
                const float z = __fdividef(vv, dd), z2 = __fmul_rn(z, z);
                return __fmul_rn(z, __fadd_rn(__fadd_rn(1.f, __fmul_rn(__fmul_rn(e2, z2), 1.f / 3.f)),
                                              __fmul_rn(__fmul_rn(__fmul_rn(e4, z2), z2), 0.2f)));
            });
        } else {
            A1[k] = pair_atan(vfma(sp(d.w), u, vmul(sp(f.x), u)), du);
            A2[k] = pair_atanh(vfma(sp(d.w), v, vmul(sp(f.x), v)), dv);
        }
    }
#pragma unroll
    for (int k = 0; k < C; ++k) {
        const float2 au = vfma(sp(f.y), A1[k], vmul(sp(f.z), A1[k]));
        const float2 av = vfma(sp(f.y), A2[k], vmul(sp(f.z), A2[k]));
        const float2 cx = vfma(au, sp(a.z), vfma(av, sp(g.x), vfma(au, sp(b.x), vmul(av, sp(g.y)))));
        const float2 cy = vfma(au, sp(a.w), vfma(av, sp(a.z), vfma(au, sp(b.y), vmul(av, sp(b.x)))));
        ax[k] = FIRST ? cx : vadd(ax[k], cx);
        ay[k] = FIRST ? cy : vadd(ay[k], cy);
    }
}

// a2-a5 for C rays (a0 ..) of node row b of the thread's two pixels, whose
// x is xc plus a node offset and whose row is at y.  Adds to acc in ray
// order; with FLAG bit 0 / 1 of near is set where a ray of the first / second
// pixel falls within the re-trace radius of a Sersic-type source.  A sum's first term is set, not added to zero.
template <int C, bool GUARD, bool FLAG, bool ODD>
__device__ __forceinline__ void pair_row(const PairSmem &sm, int nn, int a0, const float *w,
                                         float2 xc, float2 y, float2 &acc, unsigned &near)
{
    float u0[C];
#pragma unroll
    for (int k = 0; k < C; ++k) u0[k] = sm.u[GUARD ? min(a0 + k, nn - 1) : a0 + k];
    float2 ax[C], ay[C];
    int l = 0;
    const int n_lens = sm.n_lens;
    if (n_lens > 0 && (sm.lens[0] & 255) == LENSED_SIE) {
        pair_sie<C, true, ODD>(sm.cf + (sm.lens[0] >> 8), y, xc, u0, ax, ay);
        l = 1;
    } else {
#pragma unroll
        for (int k = 0; k < C; ++k) ax[k] = ay[k] = sp(0.f);
    }
    for (; l < n_lens; ++l) {
        const int e = sm.lens[l], t = e & 255;
        const float *cc = sm.cf + (e >> 8);
        if (t == LENSED_SIE) {
            pair_sie<C, false, ODD>(cc, y, xc, u0, ax, ay);
        } else if (t == LENSED_SHEAR) {
            const float4 a = reinterpret_cast<const float4 *>(cc)[0];  // -x0 -y0 g1 g2
            const float ng1 = cc[kPairNSn];
            const float2 dy = vadd(y, sp(a.y));
            const float2 g2dy = vmul(sp(a.w), dy), g1dy = vmul(sp(ng1), dy);
#pragma unroll
            for (int k = 0; k < C; ++k) {
                const float2 dx = vadd(vadd(xc, sp(u0[k])), sp(a.x));
                ax[k] = vadd(ax[k], vfma(sp(a.z), dx, g2dy));
                ay[k] = vadd(ay[k], vfma(sp(a.w), dx, g1dy));
            }
        } else {  // point mass
            const float nx0 = cc[0], ny0 = cc[1], te2 = cc[2];
            const float2 dy = vadd(y, sp(ny0)), dy2 = vmul(dy, dy);
#pragma unroll
            for (int k = 0; k < C; ++k) {
                const float2 dx = vadd(vadd(xc, sp(u0[k])), sp(nx0));
                const float2 r2 = vfma(dx, dx, dy2);
                const float2 f = vmap(r2, [=](float r) { return r > 0.f ? __fdividef(te2, r) : 0.f; });
                ax[k] = vfma(f, dx, ax[k]);
                ay[k] = vfma(f, dy, ay[k]);
            }
        }
    }
    // lens equation y = x - alpha(x)
#pragma unroll
    for (int k = 0; k < C; ++k) {
        ax[k] = vsub(vadd(xc, sp(u0[k])), ax[k]);
        ay[k] = vsub(y, ay[k]);
    }
    float2 I[C];
#pragma unroll
    for (int k = 0; k < C; ++k) I[k] = sp(0.f);
    const int n_fore = sm.n_fore, n_light = sm.n_light;
    for (int q = 0; q < n_light; ++q) {
        const float *cc = sm.cf + sm.light[q];
        const LightP L = load_light_tail(cc);
        if (L.kind == (float)kKindFlat) {
#pragma unroll
            for (int k = 0; k < C; ++k) I[k] = vadd(I[k], sp(L.A));
            continue;
        }
        const float4 a = reinterpret_cast<const float4 *>(cc)[0];
        const float csl = cc[4], snl = cc[5];
        const float2 g = reinterpret_cast<const float2 *>(cc)[kPairNSn / 2];
        if (q < n_fore) {
            const float2 dy = vadd(y, sp(a.y));
            const float2 rdu = vfma(dy, sp(a.w), vmul(dy, sp(snl)));
            const float2 rdv = vfma(dy, sp(a.z), vmul(dy, sp(csl)));
#pragma unroll
            for (int k = 0; k < C; ++k) {
                const float2 dx = vadd(vadd(xc, sp(u0[k])), sp(a.x));
                const float2 u = vfma(dx, sp(a.z), vfma(dx, sp(csl), rdu));
                const float2 v = vfma(dx, sp(g.x), vfma(dx, sp(g.y), rdv));
                float2 r2;
                I[k] = vadd(I[k], pair_light(L, u, v, r2));
            }
        } else {
            float2 even = sp(kCuspRho2), pmin = even;
#pragma unroll
            for (int k = 0; k < C; ++k) {
                const float2 dx = vadd(ax[k], sp(a.x)), dy = vadd(ay[k], sp(a.y));
                const float2 u = vfma(dx, sp(a.z), vfma(dy, sp(a.w), vfma(dx, sp(csl), vmul(dy, sp(snl)))));
                const float2 v = vfma(dy, sp(a.z), vfma(dx, sp(g.x), vfma(dy, sp(csl), vmul(dx, sp(g.y)))));
                float2 r2;
                I[k] = vadd(I[k], pair_light(L, u, v, r2));
                if (FLAG && L.kind == (float)kKindPower) {
                    // two rays at a time: three-operand minima
                    if ((k & 1) || k == C - 1)
                        pmin = make_float2(min3(pmin.x, even.x, r2.x), min3(pmin.y, even.y, r2.y));
                    even = r2;
                }
            }
            if (FLAG && L.kind == (float)kKindPower)
                near |= (pmin.x < kCuspRho2 ? 1u : 0u) | (pmin.y < kCuspRho2 ? 2u : 0u);
        }
    }
#pragma unroll
    for (int k = 0; k < C; ++k)
        if (!GUARD || a0 + k < nn) acc = vfma(sp(w[a0 + k]), I[k], acc);
}

// A rule with NN nodes per row (EXACT), its rows in chunks of at most 4 rays
// (5: 3 + 2, 6: 3 + 3, 7: 4 + 3, 8: 4 + 4), or with any number (chunks of 4,
// guarded).  5 at once measure 3 % faster on the 200x200 workload but spill
// at 80 registers; without that bound (123 registers, 4 warps per scheduler)
// they are 2 % slower than with it.
template <int NN, bool EXACT, bool FLAG>
__device__ __forceinline__ void pair_pixels(const PairSmem &sm, const SysDev &S, float2 jc,
                                            float2 ic, float2 &acc, unsigned &near)
{
    // pixel centre (j - cx) h with h as a float pair: one rounding, no
    // coherent scale error
    const float2 xc = vfma(jc, sp(S.h), vmul(jc, sp(S.h_lo)));
    const float2 yc = vfma(ic, sp(S.h), vmul(ic, sp(S.h_lo)));
    const int nn = EXACT ? NN : S.nn;
    constexpr int kChunks = EXACT ? (NN + 3) / 4 : 1;
    constexpr int C1 = EXACT ? (NN + kChunks - 1) / kChunks : 4;  // rays per chunk
    constexpr int CL = EXACT ? NN - (kChunks - 1) * C1 : 0;       // of the last one
    const float *w = sm.w;
    for (int b = 0; b < nn; ++b) {
        const float2 y = vadd(yc, sp(sm.u[b]));
        if constexpr (EXACT) {
            if constexpr (NN == 8) {
                // the two chunks of 4 share one copy of the code, the largest of
                // all: inlined twice it was slower than the one-pixel form with
                // several lenses (FP32, 91 points of 160 x 160 pixels, two lenses:
                // 1,025 us one pixel a thread, 1,074 with two copies, 1,000 with
                // one; one lens: 530, 491 and 505)
#pragma unroll 1
                for (int a0 = 0; a0 < NN; a0 += C1)
                    pair_row<C1, false, FLAG, false>(sm, nn, a0, w, xc, y, acc, near);
            } else {
                for (int a0 = 0; a0 + C1 < NN; a0 += C1)
                    pair_row<C1, false, FLAG, false>(sm, nn, a0, w, xc, y, acc, near);
                pair_row<CL, false, FLAG, (NN & 1) != 0>(sm, nn, NN - CL, w, xc, y, acc, near);
            }
            w += kPairW;
        } else {
            for (int a0 = 0; a0 < nn; a0 += C1)
                pair_row<C1, true, FLAG, false>(sm, nn, a0, w, xc, y, acc, near);
            w += nn;
        }
    }
}

}  // namespace lensed
