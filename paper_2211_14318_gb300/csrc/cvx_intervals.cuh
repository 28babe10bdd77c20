// cvx_intervals.cuh -- which parts of a rank-one line of the damage energy can
// hold a sample at or below a given level of v - s x, from the samples at the
// ends of its intervals and an upper bound of v'' (used by the lane-per-line
// scan and by the FP64 refinement's certificate).
#pragma once

#include "cvx_internal.h"

namespace cvx {

// A side of a line (its samples left or right of the centre) is cut into
// intervals of 2 PP samples.  Only their end points are sampled first.
// Inside an interval of length delta in t the function g = v - s x lies at
// most M delta^2 / 8 below the lower of its end values, M any upper bound of
// v'' there, so an interval whose bound exceeds a level holds no sample at or
// below it.
//
// Bound of v'': v = phi(d(t)) with phi' = 1 + K2' 2^{-max(d, 0)} (C ln 2 = K2')
// positive and nonincreasing, phi'' <= 0, so v'' <= phi'(min d) max(d'', 0);
//   d'' = 2 A2 + (cJ / J)^2 (c0 - c1 log2 J),
//   c0 = 2 B2 / ln2^2 - B1 / ln2, c1 = 2 B2 / ln2,
// whose positive part falls with J, so its maximum over eight intervals is
// taken at their smallest J, and d lies at most eta = max(d'') delta^2 / 8
// below its end values, which raises 2^{-d} by at most 2^eta <= 1 + eta
// (eta <= 1).  Intervals that reach J <= 0 are always kept; eight intervals
// with J <= 0 throughout hold no finite sample.
// The rounding of the samples (kEps32 max(kappa', |v| + C) bounds it, with
// |v| <= |g| + |s| m0) is covered four times over: by `base` (iv_base) and by
// the term in |e| of the comparison.
struct IvGeom {
    float h, q8;  // sample spacing, delta^2 / 8
    float rPP;    // 1 / PP
    int m0, PP;   // samples per side, pairs per interval
};

// Pairs per interval on a side of m0 samples: about sqrt(m0) samples (an end
// costs about two samples, one to two intervals per side are sampled), at
// most 32 intervals per side (one mask bit each).  0.35 / 0.5 / 0.65 / 0.8: 10.07 /
// 9.81 / 10.75 / 10.97 ms (an FE step, L = 333), 63.2 / 59.7 / 59.0 / 59.6 ms
// (a mesh, L = 1025), at L = 2049 within 2 % of each other.
constexpr float kIvScale = 0.5f;

__device__ __forceinline__ IvGeom iv_geom(float h, int m0) {
    IvGeom g;
    g.h = h;
    g.m0 = m0;
    g.PP = max(max(((m0 >> 1) + 31) >> 5, (int)(kIvScale * sqrtf((float)m0) + 0.5f)), 1);
    g.rPP = 1.0f / (float)g.PP;
    g.q8 = 0.5f * (float)(g.PP * g.PP) * h * h;
    return g;
}

// Intervals of a region of npr pairs: ceil(npr / PP).
__device__ __forceinline__ int iv_count(const IvGeom &g, int npr) {
    return (int)(((float)(npr + g.PP - 1) + 0.5f) * g.rPP);
}

__device__ __forceinline__ float iv_base(float kap, float C, float s, int m0) {
    return 4.0f * kEps32 * (kap + C + fabsf(s) * (float)m0);
}

// The constants of a line: sample_nh2's, and those of d''.
struct IvLine {
    NHPair c;
    float A2, cJ, J0, K2, c0, c1;
};

__device__ __forceinline__ IvLine iv_line(const NodeLine &nl, float A1, float A2, float cJ) {
    IvLine l;
    l.c = nh_pair_node(nl);
    l.c.A1 = pk2(A1, A1);
    l.c.A2 = pk2(A2, A2);
    l.c.CJ = pk2(cJ, cJ);
    l.J0 = nl.J0;
    l.c.J0 = pk2(l.J0, l.J0);
    l.A2 = A2;
    l.cJ = cJ;
    l.K2 = nl.K2;
    l.c1 = 2.0f * nl.B2 * (1.0f / kLn2);
    l.c0 = (l.c1 - nl.B1) * (1.0f / kLn2);
    return l;
}

// g = v - s x at two samples, and 2^{-max(d, 0)} there.
__device__ __forceinline__ void iv_eval(const NHPair &c, f32x2 H, f32x2 NS, f32x2 X, float &g0,
                                        float &g1, float &E0, float &E1) {
    const f32x2 T = mul2(X, H);
    const f32x2 P = fma2(T, fma2(T, c.A2, c.A1), c.A0);
    float j0, j1, d0, d1;
    upk2(fma2(T, c.CJ, c.J0), j0, j1);
    const f32x2 LG = pk2(lg2_approx(j0), lg2_approx(j1));
    const f32x2 D = fma2(LG, fma2(LG, c.B2, c.B1), P);
    upk2(D, d0, d1);
    const float m0 = fmaxf(d0, 0.0f), m1 = fmaxf(d1, 0.0f);
    E0 = ex2_approx(-m0);
    E1 = ex2_approx(-m1);
    upk2(fma2(NS, X, fma2(c.NK1, pk2(E0, E1), nh_branch2(c, D, m0, m1))), g0, g1);
}

// Intervals (a mask) of the region from sample xb (value ga, Ea) to fl with
// NI intervals that can hold a sample with v - s x <= e.  kLower: e follows
// the smallest end value seen (the search for the minimum), else it is fixed.
template <bool kLower>
__device__ __forceinline__ unsigned iv_sweep(const IvLine &l, const IvGeom &G, f32x2 H, f32x2 NS,
                                             float base, int xb, float fl, int NI, float ga,
                                             float Ea, float &e) {
    const float h = G.h, fS = 2.0f * (float)G.PP;
    unsigned mask = 0;
    float xa = (float)xb;  // the left end of the next interval
#pragma unroll 1
    for (int i0 = 0; i0 < NI; i0 += 8) {
        // the largest d'' over the eight intervals
        const float xe = fminf(__fmaf_rn(8.0f, fS, xa), fl);
        const float Ja = __fmaf_rn(xa * h, l.cJ, l.J0), Je = __fmaf_rn(xe * h, l.cJ, l.J0);
        const float Jm = fminf(Ja, Je);
        if (!(fmaxf(Ja, Je) > 0.0f)) {
            ga = INFINITY;
            xa = xe;
            continue;
        }
        const float r = __fdividef(l.cJ, Jm);
        const float dd =
            __fmaf_rn(r * r, fmaxf(__fmaf_rn(-l.c1, lg2_approx(Jm), l.c0), 0.0f), 2.0f * l.A2);
        float eta = dd * G.q8;
        if (!(Jm > 0.0f) || !(eta < 1e30f)) eta = INFINITY;
        const float up = eta <= 1.0f ? 1.0f + eta : INFINITY;
        const float etc = 1.0001f * eta;
        unsigned bit = 1u << i0;
        const int ie = min(i0 + 8, NI);
#pragma unroll 1
        for (int i = i0; i < ie; i += 2, bit <<= 2) {
            const float x0 = fminf(xa + fS, fl), x1 = fminf(__fmaf_rn(2.0f, fS, xa), fl);
            float p0, p1, E0, E1;
            iv_eval(l.c, H, NS, pk2(x0, x1), p0, p1, E0, E1);
            if (kLower) e = fmin3(e, p0, p1);
            // (Ea * up is NaN only where both are 0 and inf: fminf takes 1)
            const float En = fminf(fmaxf(Ea, fmaxf(E0, E1)) * up, 1.0f);
            const float thr = __fmaf_rn(etc, __fmaf_rn(l.K2, En, 1.0f), base) +
                              __fmaf_rn(4.0f * kEps32, fabsf(e), e);
            if (!(fminf(ga, p0) > thr)) mask |= bit;
            if (!(fminf(p0, p1) > thr)) mask |= bit << 1;
            ga = p1;
            Ea = E1;
            xa = x1;
        }
    }
    return mask & (NI >= 32 ? 0xffffffffu : (1u << NI) - 1u);
}

// Second derivative of v on [t0, t1]: +1 and a positive lower bound `low` of
// v'' if it is positive there, -1 if it is negative, 0 if undecided.  With E =
// 2^{-max(d, 0)}, v'' = d'' + K2' E (d'' - ln 2 d'^2 [d > 0]).  d'' lies
// between its values for the smallest and the largest J; where it is positive
// |d'| is largest at an end, and d lies at most max(d'') (t1 - t0)^2 / 8
// below its end values.  The margins (1e-4 of the terms' magnitudes, 1e-5 of
// those of d') are far above the FP32 rounding.
__device__ __forceinline__ int line_shape(const IvLine &l, float t0, float t1, float &low) {
    float A0, A1, B1, B2, u;
    upk2(l.c.A0, A0, u);
    upk2(l.c.A1, A1, u);
    upk2(l.c.B1, B1, u);
    upk2(l.c.B2, B2, u);
    const float Ja = __fmaf_rn(t0, l.cJ, l.J0), Jb = __fmaf_rn(t1, l.cJ, l.J0);
    const float Jn = fminf(Ja, Jb), Jx = fmaxf(Ja, Jb);
    if (!(Jn > 0.0f)) return 0;
    const float lga = lg2_approx(Ja), lgb = lg2_approx(Jb);
    const float lgn = fminf(lga, lgb), lgx = fmaxf(lga, lgb);
    const float cn2 = (l.cJ / Jn) * (l.cJ / Jn), cx2 = (l.cJ / Jx) * (l.cJ / Jx);
    const float fn = __fmaf_rn(-l.c1, lgn, l.c0), fx = __fmaf_rn(-l.c1, lgx, l.c0);
    const float Dx = __fmaf_rn(cn2, fmaxf(fn, 0.0f), 2.0f * l.A2);
    const float Dn = __fmaf_rn(fx >= 0.0f ? cx2 : cn2, fx, 2.0f * l.A2);
    const float Dm = __fmaf_rn(cn2, fmaxf(fabsf(fn), fabsf(fx)), 2.0f * l.A2);
    if (!(Dm < 1e30f)) return 0;
    const float da = __fmaf_rn(lga, __fmaf_rn(lga, B2, B1), __fmaf_rn(t0, __fmaf_rn(t0, l.A2, A1), A0));
    const float db = __fmaf_rn(lgb, __fmaf_rn(lgb, B2, B1), __fmaf_rn(t1, __fmaf_rn(t1, l.A2, A1), A0));
    const float ka = l.cJ / Ja * (1.0f / kLn2), kb = l.cJ / Jb * (1.0f / kLn2);
    const float ra = __fmaf_rn(2.0f * B2, lga, B1), rb = __fmaf_rn(2.0f * B2, lgb, B1);
    const float pa = __fmaf_rn(ka, ra, __fmaf_rn(2.0f * l.A2, t0, A1));
    const float pb = __fmaf_rn(kb, rb, __fmaf_rn(2.0f * l.A2, t1, A1));
    const float mg = 1e-5f * (fabsf(A1) + 2.0f * l.A2 * fmaxf(fabsf(t0), fabsf(t1)) +
                              fmaxf(fabsf(ka), fabsf(kb)) *
                                  (fabsf(B1) + 2.0f * B2 * fmaxf(fabsf(lga), fabsf(lgb))));
    const float eta = Dx * (t1 - t0) * (t1 - t0) * 0.125f;
    const float dn = fminf(da, db) - eta;
    const float Ex = dn > 0.0f ? 1.00001f * ex2_approx(-dn) : 1.0f;
    const float Ke = l.K2 * fminf(Ex, 1.0f);
    const float px = fmaxf(fabsf(pa), fabsf(pb)) + mg;
    const float qx = kLn2 * px * px;
    // v'' is linear in E: its lower bound at E = 0 or the largest E
    low = Dn + Ke * fminf(0.0f, Dn - qx) - 1e-4f * (Dm + Ke * (Dm + qx));
    if (Dn > 0.0f && low > 0.0f) return 1;
    // concave: d > 0 throughout, |d'| from below
    const float dmag = 1e-5f * (fabsf(A0) + fabsf(A1) * fmaxf(fabsf(t0), fabsf(t1)) + 1.0f);
    if (!(dn > dmag) || !(Dn > 0.0f) || !(pa * pb > 0.0f)) return 0;
    const float pn = fminf(fabsf(pa), fabsf(pb)) - mg;
    if (!(pn > 0.0f)) return 0;
    const float En = l.K2 * ex2_approx(-fmaxf(da, db)) * 0.9999f;
    const float qn = kLn2 * pn * pn;
    return Dx + En * (Dx - qn) < -1e-4f * (Dm + Ke * (Dm + qx)) ? -1 : 0;
}

}  // namespace cvx
