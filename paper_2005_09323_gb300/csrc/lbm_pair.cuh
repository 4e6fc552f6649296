// The collisions of lbm_step.cuh on pairs of sites with the packed FP32
// instructions of sm_100 and later (add, mul and fma on two floats at once).
// A packed instruction takes one issue slot for two sites, and the kernels that
// use these are bound by issue slots, not by memory: of the 169 instructions
// per site and step of the register-staged FP32 kernel about 90 are this
// arithmetic.
//
// Every result is the same bits as the scalar collision's: the packed forms
// round each half as the scalar instructions do, and the fused multiply-adds
// below are the ones the compiler forms from the scalar expressions.  A compiler
// that formed others would show where every variant of the step is run from one
// random state far from equilibrium (tests/test_gpu_packed.py: both collisions,
// periodic with force, open with varying rates, three storage formats).
#pragma once
#include "lbm_device.cuh"
#include "step_params.h"

namespace lbm {

__device__ __forceinline__ float2 splat(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, splat(-1.0f), a); }   // a - b

// 1 / x of a density (1 plus an FP32 number: 0 or at least 2^-24 in magnitude)
__device__ __forceinline__ float rcp_density(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float2 rcp_density2(float2 x) { return make_float2(rcp_density(x.x), rcp_density(x.y)); }

// one opposite pair of directions (bgk_pair)
template <bool FORCE>
__device__ __forceinline__ void bgk_pair2(float2& gq, float2& go, float2 cu, float A, float B, float wq, float2 P,
                                          float2 Qc, float2 a0, float2 omm)
{
    const float2 E = fma2(cu, FORCE ? fma2(Qc, cu, splat(A)) : fma2(Qc, cu, splat(0.0f)), a0);
    const float2 O = fma2(P, cu, FORCE ? splat(B) : splat(0.0f));
    gq = fma2(splat(wq), add2(E, O), mul2(omm, gq));
    go = fma2(splat(wq), sub2(E, O), mul2(omm, go));
}

// bgk_collide of the pair of sites i
template <int N, bool FORCE>
__device__ __forceinline__ void bgk_collide2(float2 (&g)[9][N], int i, const BgkConsts& k, float2 om)
{
    const float2 s1 = add2(g[1][i], g[3][i]), d1 = sub2(g[1][i], g[3][i]);
    const float2 s2 = add2(g[2][i], g[4][i]), d2 = sub2(g[2][i], g[4][i]);
    const float2 s5 = add2(g[5][i], g[7][i]), d5 = sub2(g[5][i], g[7][i]);
    const float2 s6 = add2(g[6][i], g[8][i]), d6 = sub2(g[6][i], g[8][i]);
    const float2 drho = add2(add2(g[0][i], s1), add2(s2, add2(s5, s6)));
    const float2 jx = add2(d1, sub2(d5, d6)), jy = add2(d2, add2(d5, d6));
    const float2 inv = rcp_density2(add2(splat(1.0f), drho));
    const float2 ux = mul2(FORCE ? add2(jx, splat(k.hgx)) : jx, inv);
    const float2 uy = mul2(FORCE ? add2(jy, splat(k.hgy)) : jy, inv);
    const float2 om3 = FORCE ? splat(k.om3) : mul2(splat(3.0f), om);
    const float2 omm = FORCE ? splat(k.omm) : sub2(splat(1.0f), om);
    const float2 P = fma2(om3, drho, om3);  // 3 om rho
    const float2 Qc = mul2(splat(1.5f), P);  // 4.5 om rho
    const float2 u2 = fma2(ux, ux, mul2(uy, uy));
    float2 a0 = fma2(om, drho, mul2(mul2(splat(-0.5f), P), u2));
    if constexpr (FORCE) a0 = fma2(splat(-k.kgx), ux, fma2(splat(-k.kgy), uy, a0));
    g[0][i] = fma2(splat(wf(0)), a0, mul2(omm, g[0][i]));
    bgk_pair2<FORCE>(g[1][i], g[3][i], ux, k.A[0], k.B[0], wf(1), P, Qc, a0, omm);
    bgk_pair2<FORCE>(g[2][i], g[4][i], uy, k.A[1], k.B[1], wf(2), P, Qc, a0, omm);
    bgk_pair2<FORCE>(g[5][i], g[7][i], add2(ux, uy), k.A[2], k.B[2], wf(5), P, Qc, a0, omm);
    bgk_pair2<FORCE>(g[6][i], g[8][i], sub2(uy, ux), k.A[3], k.B[3], wf(6), P, Qc, a0, omm);
}

// cm_collide of the pair of sites i; ws, a, b: the shear rate and the k20, k02
// block of Omega
template <int N, bool FORCE>
__device__ __forceinline__ void cm_collide2(float2 (&g)[9][N], int i, const BgkConsts& k, const CmConsts& m, float2 ws,
                                            float2 a, float2 b)
{
    const float2 s1 = add2(g[1][i], g[3][i]), d1 = sub2(g[1][i], g[3][i]);
    const float2 s2 = add2(g[2][i], g[4][i]), d2 = sub2(g[2][i], g[4][i]);
    const float2 s5 = add2(g[5][i], g[7][i]), d5 = sub2(g[5][i], g[7][i]);
    const float2 s6 = add2(g[6][i], g[8][i]), d6 = sub2(g[6][i], g[8][i]);
    const float2 drho = add2(add2(g[0][i], s1), add2(s2, add2(s5, s6)));
    const float2 jx = add2(d1, sub2(d5, d6)), jy = add2(d2, add2(d5, d6));
    const float2 rho = add2(splat(1.0f), drho);
    const float2 inv = rcp_density2(rho);
    const float2 m22 = add2(s5, s6), m20 = add2(s1, m22), m02 = add2(s2, m22), m11 = sub2(s5, s6), m21 = add2(d5, d6),
                 m12 = sub2(d5, d6);
    const float2 ux = mul2(FORCE ? add2(jx, splat(k.hgx)) : jx, inv);
    const float2 uy = mul2(FORCE ? add2(jy, splat(k.hgy)) : jy, inv);
    const float2 fx = splat(m.fx), fy = splat(m.fy);
    // negated: the moments subtract these products
    const float2 nux = mul2(splat(-1.0f), ux), nuy = mul2(splat(-1.0f), uy), nrux = mul2(rho, nux), nruy = mul2(rho, nuy);
    float2 M20 = fma2(nrux, ux, fma2(splat(-(1.0f / 3.0f)), drho, m20));
    float2 M02 = fma2(nruy, uy, fma2(splat(-(1.0f / 3.0f)), drho, m02));
    float2 M11 = fma2(nrux, uy, m11);
    float2 M21 = fma2(nruy, splat(1.0f / 3.0f), m21);
    float2 M12 = fma2(nrux, splat(1.0f / 3.0f), m12);
    float2 M22 = fma2(fma2(nrux, ux, mul2(nruy, uy)), splat(1.0f / 3.0f), fma2(splat(-(1.0f / 9.0f)), drho, m22));
    float2 uF = splat(0.0f);
    if constexpr (FORCE) {
        uF = fma2(ux, fx, mul2(uy, fy));
        M20 = fma2(ux, fx, M20);
        M02 = fma2(uy, fy, M02);
        M11 = fma2(splat(0.5f), fma2(ux, fy, mul2(uy, fx)), M11);
        M21 = fma2(fy, splat(1.0f / 6.0f), M21);
        M12 = fma2(fx, splat(1.0f / 6.0f), M12);
        M22 = fma2(uF, splat(1.0f / 3.0f), M22);
    }
    const float2 u2x = add2(ux, ux), u2y = add2(uy, uy), n2x = add2(nux, nux), n2y = add2(nuy, nuy);
    const float2 uxx = mul2(ux, ux), uyy = mul2(uy, uy), uxy = mul2(add2(u2x, u2x), uy);
    // central moments, relaxed
    const float2 k21 = fma2(nuy, M20, fma2(n2x, M11, M21));
    const float2 k12 = fma2(nux, M02, fma2(n2y, M11, M12));
    const float2 k22 = fma2(uxy, M11, fma2(uyy, M20, fma2(uxx, M02, fma2(n2y, M21, fma2(n2x, M12, M22)))));
    const float2 r20 = fma2(a, M20, mul2(b, M02)), r02 = fma2(b, M20, mul2(a, M02)), r11 = mul2(ws, M11);
    const float2 r21 = mul2(splat(m.w3), k21), r12 = mul2(splat(m.w3), k12), r22 = mul2(splat(m.w4), k22);
    // back to raw moments
    const float2 R21 = fma2(uy, r20, fma2(u2x, r11, r21));
    const float2 R12 = fma2(ux, r02, fma2(u2y, r11, r12));
    const float2 R22 = fma2(uxy, r11, fma2(uyy, r20, fma2(uxx, r02, fma2(u2y, r21, fma2(u2x, r12, r22)))));
    if constexpr (FORCE) {
        // Guo term
        const float2 t0 = mul2(splat(-3.0f), uF);
        const float2 c5 = add2(ux, uy), f5 = add2(fx, fy), c6 = sub2(uy, ux), f6 = sub2(fy, fx);
        const float2 e1 = fma2(mul2(splat(9.0f), ux), fx, t0), e2 = fma2(mul2(splat(9.0f), uy), fy, t0);
        const float2 e5 = fma2(mul2(splat(9.0f), c5), f5, t0), e6 = fma2(mul2(splat(9.0f), c6), f6, t0);
        auto guo = [&](int q, float2 e, float2 f, float s) { g[q][i] = fma2(splat(wf(q)), fma2(splat(s), f, e), g[q][i]); };
        g[0][i] = fma2(splat(wf(0)), t0, g[0][i]);
        guo(1, e1, fx, 3.0f);
        guo(3, e1, fx, -3.0f);
        guo(2, e2, fy, 3.0f);
        guo(4, e2, fy, -3.0f);
        guo(5, e5, f5, 3.0f);
        guo(7, e5, f5, -3.0f);
        guo(6, e6, f6, 3.0f);
        guo(8, e6, f6, -3.0f);
    }
    g[0][i] = sub2(g[0][i], sub2(sub2(R22, r20), r02));
    g[1][i] = fma2(splat(-0.5f), sub2(sub2(r20, R12), R22), g[1][i]);
    g[3][i] = fma2(splat(-0.5f), sub2(add2(r20, R12), R22), g[3][i]);
    g[2][i] = fma2(splat(-0.5f), sub2(sub2(r02, R21), R22), g[2][i]);
    g[4][i] = fma2(splat(-0.5f), sub2(add2(r02, R21), R22), g[4][i]);
    const float2 p5 = add2(r11, R21), m5 = sub2(r11, R21);  // -r11 + R21 and -r11 - R21 are their negatives
    g[5][i] = fma2(splat(-0.25f), add2(add2(p5, R12), R22), g[5][i]);
    g[7][i] = fma2(splat(-0.25f), add2(sub2(m5, R12), R22), g[7][i]);
    g[6][i] = fma2(splat(-0.25f), sub2(R22, add2(m5, R12)), g[6][i]);
    g[8][i] = fma2(splat(-0.25f), add2(sub2(R12, p5), R22), g[8][i]);
}

// the periodic channel's collision of the pair of sites i
template <int COLL, int N>
__device__ __forceinline__ void collide_pair(float2 (&g)[9][N], int i, const StepParams& p)
{
    if constexpr (COLL == 0)
        bgk_collide2<N, true>(g, i, p.bgk, splat(p.bgk.om));
    else
        cm_collide2<N, true>(g, i, p.bgk, p.cm, splat(p.cm.ws), splat(p.cm.a), splat(p.cm.b));
}

template <int COLL, int N>
__device__ __forceinline__ void collide2(float2 (&g)[9][N], const StepParams& p)
{
#pragma unroll
    for (int i = 0; i < N; ++i) collide_pair<COLL>(g, i, p);
}

// f(pairs, i) on every pair of the V sites of g
template <int V, typename F>
__device__ __forceinline__ void on_pairs(float (&g)[9][V], F&& f)
{
    float2 h[9][V / 2];
#pragma unroll
    for (int q = 0; q < 9; ++q)
#pragma unroll
        for (int i = 0; i < V / 2; ++i) h[q][i] = make_float2(g[q][2 * i], g[q][2 * i + 1]);
#pragma unroll
    for (int i = 0; i < V / 2; ++i) f(h, i);
#pragma unroll
    for (int q = 0; q < 9; ++q)
#pragma unroll
        for (int i = 0; i < V / 2; ++i) {
            g[q][2 * i] = h[q][i].x;
            g[q][2 * i + 1] = h[q][i].y;
        }
}

// the open channel's collision of the pair of sites i at the rates om
template <int COLL, int N>
__device__ __forceinline__ void collide_at2(float2 (&g)[9][N], int i, const StepParams& p, float2 om)
{
    if constexpr (COLL == 0) {
        bgk_collide2<N, false>(g, i, p.bgk, om);
    } else {
        const float2 wb = splat(p.cm.wb);
        cm_collide2<N, false>(g, i, p.bgk, p.cm, om, mul2(splat(0.5f), add2(wb, om)),
                              mul2(splat(0.5f), sub2(wb, om)));
    }
}

}  // namespace lbm
