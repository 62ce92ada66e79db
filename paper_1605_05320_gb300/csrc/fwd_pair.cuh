// fwd_pair.cuh -- FP32 edge arithmetic of the forward step (Sec. 6: Roe-type
// f-wave solver for the shallow water equations with bathymetry; the
// wave-propagation update with MC-limited corrections), shared by the
// single-grid strips, the patch strips, the refluxing fluxes and the 1D step.
//
// Every operation rounds as written (__fadd_rn/__fmul_rn, which the
// compiler never fuses, explicit fmaf, and .rn packed operations), so an
// edge gets the same bits whichever kernel computes it and whichever edges
// share its warp.
//
// The update is branch-free.  A wave of speed s goes right with weight
// (1 + sign s)/2 (1, 1/2 at s = 0, 0) and left with the rest, so the
// fluctuations are A+dQ = sum (1 + sign s^p)/2 Z^p and A-dQ the rest (an
// f-wave of speed 0 is split half and half).  The MC-limited correction
// needs no division by the wave norm: for Z = b (1, s, vhat) and its upwind
// neighbour Zu = bu (1, su, vu), theta b = bu (1 + su s + vu vhat) /
// (1 + s^2 + vhat^2), and phi(theta) b is formed from b and theta b alone
// (zero when b = 0).  A warp whose edges are all subsonic (s1 < 0 < s3)
// takes the SUB form, which drops the operations whose outcome that fixes
// (weights 0 and 1, upwind sides, signs); it gives the same numbers as the
// general form, up to the sign of an exact zero.
//
// What bounds these kernels is the number of instructions issued, and waves 1
// and 3 of an edge take the same operations, so the SUB form and the solve
// run the two as the halves of packed FP32x2 instructions: a packed
// operation occupies the FMA pipe twice but issues once, and each half
// rounds like the scalar operation.
// 4096^2 with waves everywhere: 256 us per step with scalar operations, 231
// to 235 us so.
#pragma once
#include "packed.cuh"

namespace swadj {
namespace fp {

__device__ __forceinline__ float fma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float fms(float a, float b, float c) { return fmaf(a, b, -c); }   // ab - c
__device__ __forceinline__ float fnma(float a, float b, float c) { return fmaf(-a, b, c); }  // c - ab
__device__ __forceinline__ float rcp(float x) { return rcp_ftz(x); }
__device__ __forceinline__ float rsq(float x) { return rsqrt_ftz(x); }

// sign(s) in {-1, 0, 1}
__device__ __forceinline__ float sgn(float s) { return s > 0.f ? 1.f : (s < 0.f ? -1.f : 0.f); }
// s > 0 ? a : b
__device__ __forceinline__ float pick(float s, float a, float b) { return s > 0.f ? a : b; }
__device__ __forceinline__ bool subsonic(float s1, float s3) { return s1 < 0.f && s3 > 0.f; }

// Half the MC-limited wave strength: phi(theta) b / 2 for the MC limiter
// phi = max(0, min((1 + theta)/2, 2, 2 theta)), given b and r = theta b: (b +
// r)/4 limited to [-m, m], m = min(|b|, |r|) where b and r have one sign and
// 0 where they do not.  The factor 1/2 is exact, so twice this is the
// limited strength to the last bit.
__device__ __forceinline__ float mc_clamp(float t, float b, float r) {
    const float m = fmaxf(min_xorsign(b, r), 0.f);
    return fmaxf(fminf(t, m), -m);
}
__device__ __forceinline__ float mch(float b, float r) {
    return mc_clamp(mul(0.25f, add(b, r)), b, r);
}
__device__ __forceinline__ f2 mch(f2 b, f2 r) {
    const f2 t = mul(dup(0.25f), add(b, r));
    return mk(mc_clamp(t.x, b.x, r.x), mc_clamp(t.y, b.y, r.y));
}

// ------------------------------------------------------------------ records
// A cell in the frame of a sweep (mn the momentum normal to the edges, mt
// the tangential one) with the data its edges need: sqrt(h), sqrt(h) times
// the normal and tangential velocity (mn / sqrt(h), mt / sqrt(h)), the
// normal momentum flux mn^2 / h and the cross flux mn mt / h.
struct Cell {
    float h, mn, mt, sq, su, sv, P, T, eta;
};

// Waves of one edge: speeds s1 = uh - ch, s3 = uh + ch (and uh of the shear
// wave), the tangential Roe velocity and the strengths of the waves
// b1 (1, s1, vh), b2 (0, 0, 1), b3 (1, s3, vh); hr = 1 / (2 ch).
struct Edge {
    float s1, s3, vh, b1, b2, b3, uh, ch, hr;
};

// The upwind neighbour of wave 1 or 3 for the limiter: its speed, tangential
// Roe velocity and strength.
struct Up {
    float s, vh, b;
};

// Net fluxes of an edge: L into the left (lower) cell, R into the right
// (upper) cell, in the edge's frame (Q -= nu * net).
struct Net {
    float L0, L1, L2, R0, R1, R2;
};

// Cell data in the frame of a sweep from (eta, h, mn, mt).
__device__ __forceinline__ Cell derive(float eta, float h, float mn, float mt) {
    const float q = rsq(h);
    Cell c;
    c.h = h; c.mn = mn; c.mt = mt; c.eta = eta;
    c.sq = mul(h, q);
    const f2 s = mul(mk(mn, mt), dup(q));
    const f2 p = mul(dup(s.x), s);
    c.su = s.x; c.sv = s.y;
    c.P = p.x; c.T = p.y;
    return c;
}

// Roe f-wave decomposition (Sec. 6 solver): hhat = (hL + hR)/2, uhat and
// vhat sqrt(h)-weighted ((sqrt(hL) uL + sqrt(hR) uR) / (sqrt(hL) +
// sqrt(hR))), chat = sqrt(g hhat); the momentum jump carries the bathymetry
// source as g hhat (etaR - etaL), so the ocean at rest has no waves.
// 1 / (s3 - s1) = 1 / (2 chat) comes from the same rsqrt as chat, or, RCP (the
// unsplit step), from a reciprocal of s3 - s1, with which the waves' momenta
// add up to the jump to one rounding.
template <bool RCP = false>
__device__ __forceinline__ Edge solve(float g_half, const Cell &L, const Cell &R) {
    Edge w;
    const float gh = mul(g_half, add(L.h, R.h));   // g hhat
    const float rd = rcp(add(L.sq, R.sq));
    const f2 uv = mul(add(mk(L.su, L.sv), mk(R.su, R.sv)), dup(rd));
    w.uh = uv.x;
    w.vh = uv.y;
    const float rc = rsq(gh);
    w.ch = mul(gh, rc);
    w.s1 = sub(w.uh, w.ch);
    w.s3 = add(w.uh, w.ch);
    const float df1 = sub(R.mn, L.mn);
    const f2 dPT = fma(mk(L.P, L.T), dup(-1.f), mk(R.P, R.T));
    const float df2 = fma(gh, sub(R.eta, L.eta), dPT.x);
    w.hr = RCP ? rcp(sub(w.s3, w.s1)) : mul(0.5f, rc);
    const f2 b = mul(mk(fms(w.s3, df1, df2), fnma(w.s1, df1, df2)), dup(w.hr));
    w.b1 = b.x;
    w.b3 = b.y;
    w.b2 = fnma(w.vh, df1, dPT.y);
    return w;
}

// Fluctuations of an edge as pairs (A-dQ, A+dQ), one per component.  A wave
// of speed s goes right with weight (1 + sign s)/2 (half each way at s = 0).
// SUB: the edge is subsonic (s1 < 0 < s3), so wave 1 goes left and wave 3
// right.
struct Fluct {
    f2 a0, a1, a2;
};
template <bool SUB>
__device__ __forceinline__ Fluct fluct(const Edge &w) {
    Fluct f;
    if (SUB) {
        f.a0 = mk(w.b1, w.b3);
        f.a1 = mul(f.a0, mk(w.s1, w.s3));
    } else {
        const float p1 = mul(fma(0.5f, sgn(w.s1), 0.5f), w.b1);
        const float p3 = mul(fma(0.5f, sgn(w.s3), 0.5f), w.b3);
        const float e1 = sub(w.b1, p1), e3 = sub(w.b3, p3);
        f.a0 = mk(add(e1, e3), add(p1, p3));
        f.a1 = mk(fma(e1, w.s1, mul(e3, w.s3)), fma(p1, w.s1, mul(p3, w.s3)));
    }
    const float p2 = mul(fma(0.5f, sgn(w.uh), 0.5f), w.b2);
    f.a2 = fma(f.a0, dup(w.vh), mk(sub(w.b2, p2), p2));
    return f;
}

// Fluctuations and MC-limited correction of edge w: L = A-dQ + F into the
// left cell, R = A+dQ - F into the right cell.  F = sum_p sign(s^p)/2 (1 - nu
// |s^p|) phi(theta^p) Z^p, computed as (sign(s) - nu s) times half the limited
// strength (the same number).  u1, u3: the upwind neighbours of waves 1 and
// 3 (the left edge for s > 0, the right one otherwise); b2l, b2r: the
// shear-wave strengths of the left and right edges.
template <bool SUB>
__device__ __forceinline__ Net net(const Edge &w, const Up &u1, const Up &u3, float b2l,
                                   float b2r, float nu, int order, const Fluct &f) {
    f2 a0 = f.a0, a1 = f.a1, a2 = f.a2;
    Net n;
    if (order >= 2) {
        const float g2 = sgn(w.uh);
        const f2 s = mk(w.s1, w.s3), b = mk(w.b1, w.b3);
        const f2 k = SUB ? fma(mk(nu, -nu), s, dup(1.f))   // sign(s) - nu s of (-wave 1, wave 3)
                         : mk(-fnma(nu, w.s1, sgn(w.s1)), fnma(nu, w.s3, sgn(w.s3)));
        // theta^p b^p = b_up (1 + s_up s + v_up vhat) / (1 + s^2 + vhat^2)
        const f2 m = fma(s, s, dup(fma(w.vh, w.vh, 1.f)));
        const f2 d = fma(mk(u1.s, u3.s), s, fma(mk(u1.vh, u3.vh), dup(w.vh), dup(1.f)));
        const f2 c = mul(k, mch(b, mul(mul(mk(u1.b, u3.b), d), rcp(m))));   // (-wave 1, wave 3)
        const float l2 = mch(w.b2, pick(w.uh, b2l, b2r));
        const float c2 = mul(fnma(nu, w.uh, g2), l2);
        const float F0 = sub(c.y, c.x);
        const float F1 = fma(-c.x, w.s1, mul(c.y, w.s3));
        const float F2 = fma(F0, w.vh, c2);
        const f2 lr = mk(1.f, -1.f);
        a0 = fma(dup(F0), lr, a0);
        a1 = fma(dup(F1), lr, a1);
        a2 = fma(dup(F2), lr, a2);
    }
    n.L0 = a0.x; n.L1 = a1.x; n.L2 = a2.x;
    n.R0 = a0.y; n.R1 = a1.y; n.R2 = a2.y;
    return n;
}

// Upwind neighbours of an edge from its left (wl) and right (wr) edges.
__device__ __forceinline__ void upwind(const Edge &w, const Edge &wl, const Edge &wr, Up &u1,
                                       Up &u3) {
    u1.s = pick(w.s1, wl.s1, wr.s1); u1.vh = pick(w.s1, wl.vh, wr.vh);
    u1.b = pick(w.s1, wl.b1, wr.b1);
    u3.s = pick(w.s3, wl.s3, wr.s3); u3.vh = pick(w.s3, wl.vh, wr.vh);
    u3.b = pick(w.s3, wl.b3, wr.b3);
}

// Net fluxes of the middle edge of three consecutive edges held by one
// thread (1D step, y-sweeps): the form is SUB when `all_sub`.
__device__ __forceinline__ Net net3(const Edge &wl, const Edge &w, const Edge &wr, float nu,
                                    int order, bool all_sub) {
    Up u1, u3;
    if (all_sub) {
        u1.s = wr.s1; u1.vh = wr.vh; u1.b = wr.b1;
        u3.s = wl.s3; u3.vh = wl.vh; u3.b = wl.b3;
        return net<true>(w, u1, u3, wl.b2, wr.b2, nu, order, fluct<true>(w));
    }
    upwind(w, wl, wr, u1, u3);
    return net<false>(w, u1, u3, wl.b2, wr.b2, nu, order, fluct<false>(w));
}

}  // namespace fp
}  // namespace swadj
