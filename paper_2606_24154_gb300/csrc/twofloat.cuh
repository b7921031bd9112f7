// twofloat.cuh -- two-float ("double-float") arithmetic on the FP32 pipe, shared by the
// mixed-precision fill (fill_mixed.cu) and the refined point evaluation (eval_acc.cu).
// Every quantity is an unevaluated sum hi + lo of two floats; sums and products keep
// their rounding errors through error-free transformations (Knuth TwoSum, FMA-based
// TwoProd), about 44 significant bits.
#pragma once
#include "eval_blocks.cuh"

namespace nb {

// All operations are the explicitly rounded intrinsics, so no contraction or reordering
// can change the error-free transformations.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& t) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    t = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
    p = __fmul_rn(a, b);
    e = __fmaf_rn(a, b, -p);
}

// (ah + al) - (bh + bl), unnormalised
__device__ __forceinline__ void df_sub(float ah, float al, float bh, float bl, float& h, float& l) {
    float t;
    two_sum(ah, -bh, h, t);
    l = __fadd_rn(t, __fsub_rn(al, bl));
}

// a . b for three-vectors of two-float components
__device__ __forceinline__ void df_dot3(const float (&ah)[3], const float (&al)[3], const float4& bh, const float4& bl,
                                        float& h, float& l) {
    float p0, e0, p1, e1, p2, e2, t1, t2, s;
    two_prod(ah[0], bh.x, p0, e0);
    two_prod(ah[1], bh.y, p1, e1);
    two_prod(ah[2], bh.z, p2, e2);
    two_sum(p0, p1, s, t1);
    two_sum(s, p2, h, t2);
    float lo = __fadd_rn(__fadd_rn(e0, e1), __fadd_rn(e2, __fadd_rn(t1, t2)));
    lo = __fmaf_rn(ah[0], bl.x, lo);
    lo = __fmaf_rn(al[0], bh.x, lo);
    lo = __fmaf_rn(ah[1], bl.y, lo);
    lo = __fmaf_rn(al[1], bh.y, lo);
    lo = __fmaf_rn(ah[2], bl.z, lo);
    lo = __fmaf_rn(al[2], bh.z, lo);
    l = lo;
}

// squared norm of (X, Y, Z), two-float components
__device__ __forceinline__ void df_norm2(float xh, float xl, float yh, float yl, float zh, float zl, float& h,
                                         float& l) {
    float px, ex, py, ey, pz, ez, s, t1, t2;
    two_prod(xh, xh, px, ex);
    two_prod(yh, yh, py, ey);
    two_prod(zh, zh, pz, ez);
    ex = __fmaf_rn(__fadd_rn(xh, xh), xl, ex);
    ey = __fmaf_rn(__fadd_rn(yh, yh), yl, ey);
    ez = __fmaf_rn(__fadd_rn(zh, zh), zl, ez);
    two_sum(px, py, s, t1);
    two_sum(s, pz, h, t2);
    l = __fadd_rn(__fadd_rn(ex, ey), __fadd_rn(ez, __fadd_rn(t1, t2)));
}

// ---------------------------------------------------------------- packed two-float nodes
// Two Gauss nodes per instruction in the packed FP32x2 forms (__fadd2_rn, __fmul2_rn,
// __ffma2_rn; a - b as fma(b, -1, a), exact like a subtraction).  Error terms of products
// come out negated, e_neg = fma(-a, b, a b) = -(a b - fl(a b)), so that no extra negation is
// needed; the running sum keeps its low part negated as well (NL = -lo).
__device__ __forceinline__ float2 bc2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2& s, float2& t) {
    s = __fadd2_rn(a, b);
    const float2 bb = sub2(s, a);
    t = __fadd2_rn(sub2(a, sub2(s, bb)), sub2(b, bb));
}

// Per-image quantities of one pair in the column element's frame, broadcast to both lanes
// (negated copies for the error terms of products).
struct PairDF2 {
    float2 xh, nxh, xl, zh, nzh, zl;  // X, Z
    float2 d2h, d2l;                  // |D|^2
};
struct NormDF2 {
    float2 nxh, nnxh, nxl, nzh, nnzh, nzl;  // local components of the row normal (x, z)
    float2 ndh, ndl;                        // n_i . D
};

// r^2 = |D|^2 + 2 (X s_x + Z s_z) + |s|^2 and 1/r for a node pair: y0 (MUFU estimate), the
// Newton correction negated (nyl = -yl), y0^2 = a exactly with its negated error nae.
__device__ __forceinline__ void node_rinv2(const PairDF2& P, const float4& q0, const float4& q1, const float4& q2,
                                           const float4& q3, float2& y0, float2& ny0, float2& nyl, float2& a,
                                           float2& na, float2& nae) {
    const float2 m1 = bc2(-1.f);
    const float2 sx = make_float2(q0.x, q0.y), sz = make_float2(q0.z, q0.w);
    const float2 s2 = make_float2(q1.x, q1.y);
    const float2 sxl = make_float2(q2.x, q2.y), szl = make_float2(q2.z, q2.w);
    const float2 s2l = make_float2(q3.x, q3.y);
    const float2 p1 = __fmul2_rn(P.xh, sx), ne1 = __ffma2_rn(P.nxh, sx, p1);
    const float2 p2 = __fmul2_rn(P.zh, sz), ne2 = __ffma2_rn(P.nzh, sz, p2);
    float2 qh, t, t2;
    two_sum2(p1, p2, qh, t);
    float2 lo = __ffma2_rn(ne1, m1, t);
    lo = __ffma2_rn(ne2, m1, lo);
    lo = __ffma2_rn(P.xh, sxl, lo);
    lo = __ffma2_rn(P.xl, sx, lo);
    lo = __ffma2_rn(P.zh, szl, lo);
    lo = __ffma2_rn(P.zl, sz, lo);
    two_sum2(qh, s2, qh, t2);
    lo = __fadd2_rn(lo, __fadd2_rn(t2, s2l));
    // |D|^2 >= |q| for d >= kFillRatioC rho (|q| <= 2 d rho + rho^2)
    const float2 r2h = __fadd2_rn(P.d2h, qh);
    const float2 t3 = sub2(qh, sub2(r2h, P.d2h));
    const float2 r2l = __fadd2_rn(P.d2l, __fadd2_rn(lo, t3));
    y0 = make_float2(rsqrtf(r2h.x), rsqrtf(r2h.y));
    ny0 = __fmul2_rn(y0, m1);
    a = __fmul2_rn(y0, y0);
    nae = __ffma2_rn(ny0, y0, a);  // a - y0^2
    na = __fmul2_rn(ny0, y0);
    const float2 b = __fmul2_rn(r2h, a);
    const float2 nbe = __ffma2_rn(r2h, na, b);  // b - r2h a
    // h = 1 - r^2 y0^2 (1 - b is exact: b within 2^-20 of 1)
    float2 h = __ffma2_rn(b, m1, bc2(1.f));
    h = __fadd2_rn(h, nbe);
    h = __ffma2_rn(r2h, nae, h);
    h = __ffma2_rn(r2l, na, h);
    nyl = __fmul2_rn(__fmul2_rn(bc2(-0.5f), y0), h);
}

// ---------------------------------------------------------------- far pairs by moments
// A pair far from its element (d >= kMomRatio radii) by the element's planar moments about its
// centroid, two images per packed instruction.  With n = D / d, y = 1 / d,
//   Phi' = A y + y^3 rho^2 (f2 + s f3 + s^2 f4),
//   E' = A D y^3 + y^3 s rho [(r2 + s r3 + s^2 r4) n - (w2 + s w3 + s^2 w4)],   s = y rho,
// the monopole and the terms of degree 2 to 4 of the multipole series of 1 / |D - u| over the
// element's points u (degree 1 vanishes about the centroid).  Only the monopole needs two-float
// arithmetic: the rest is below (rho / d)^2 / 5 of the pair, so plain FP32 leaves an error of about
// 1e-7 of that (1e-11 of the pair at 64 radii).  190 FP32 lane operations per pair for Phi' and E' (124
// for Phi' alone) and one MUFU root, where four Gauss nodes in two-float arithmetic took 549
// (283) and four roots, six 743 and nine 1131.  What the series leaves out (odd moments of a
// triangle: degree 5) is 2.8e-9 of the pair at 24 radii, where the 6-point rule has 1.9e-9, 1.3e-9 at
// kMomRatio = 28, and 2e-11 at 64 radii, where the 4-point rules have 3e-9 (worst over triangles,
// slivers, 10:1 strips and skewed quadrilaterals, 400 directions).
// ElemMom per element: every constant twice (both lanes), two constants per float4:
//   3 M20, 3 M11 | 3 M02, -t2 / 2 | k30, k21 | k12, k03 | -tx, -tz | K40, K31 | K13, K04 | T31, T22 | T13, P20 |
//   P11, P02 | q0, 5 q0 | -3 t2 / 2, then the area A as hi, lo
// with M the moments of u = (node - centroid) / rho in the element plane (scaled by the element's radius, so
// that they are FP32 numbers at any size of the geometry), t2 = M20 + M02, k = 7.5 M, (tx, tz) = 1.5
// (M30 + M12, M21 + M03), K = 17.5 M, T = 3 K, P = -7.5 (M40 + M22, M31 + M13, M22 + M04), q0 = 0.375 (M40 +
// 2 M22 + M04).
constexpr double kMomRatio = 28.0;
constexpr int kMomF4 = 12;

struct MomSum2 {  // sums over the images of an element, both lanes
    float2 ph, pl;                        // y, two floats (times A: the monopole's potential)
    float2 xh, xl, yh, yl, zh, zl;        // D y^3, two floats: minus the high part, the low part
    float2 fc, ex, ey, ez;                // the other terms, FP32, over rho^2 and rho
};

__device__ __forceinline__ float2 lane2(const float4& v, int i) {
    return i ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
}

// One step: local differences X, Y, Z (two floats each) of two images; lanes with far = false add 0.
// Returns nothing for them: the caller evaluates those pairs itself.  d2h is |D|^2's high part.
template <bool kPhi, bool kField>
__device__ __forceinline__ void mom_pair2(const float4* __restrict__ mom, float rho, float2 xh, float2 xl, float2 yh, float2 yl,
                                          float2 zh, float2 zl, float2 d2h, float2 d2l, bool far0, bool far1,
                                          MomSum2& S) {
    const float2 m1 = bc2(-1.f);
    const float2 y0 = make_float2(far0 ? rsqrtf(d2h.x) : 0.f, far1 ? rsqrtf(d2h.y) : 0.f);
    // y = y0 + ye: one Newton step in two floats (h = 1 - d2 y0^2)
    const float2 ny0 = __fmul2_rn(y0, m1);
    const float2 a = __fmul2_rn(y0, y0), na = __fmul2_rn(ny0, y0);
    const float2 nae = __ffma2_rn(ny0, y0, a);  // a - y0^2
    const float2 b = __fmul2_rn(d2h, a);
    const float2 nbe = __ffma2_rn(d2h, na, b);
    float2 h = __ffma2_rn(b, m1, bc2(1.f));
    h = __fadd2_rn(h, nbe);
    h = __ffma2_rn(d2h, nae, h);
    h = __ffma2_rn(d2l, na, h);
    // a lane that is not far has y0 = 0, so h = 1 and ye = 0
    const float2 ye = __fmul2_rn(__fmul2_rn(bc2(0.5f), y0), h);
    float2 t;
    if constexpr (kPhi) {
        two_sum2(S.ph, y0, S.ph, t);
        S.pl = __fadd2_rn(S.pl, __fadd2_rn(t, ye));
    }
    const float2 c3 = __fmul2_rn(a, y0);
    if constexpr (kField) {
        // y^3 = c3 + cl, y^2 = a + (2 y0 ye - nae)
        const float2 y2l = __ffma2_rn(nae, m1, __fmul2_rn(__fadd2_rn(y0, y0), ye));
        const float2 nc3 = __fmul2_rn(na, y0);
        float2 cl = __ffma2_rn(a, y0, nc3);
        cl = __ffma2_rn(a, ye, cl);
        cl = __ffma2_rn(y2l, y0, cl);
        auto add = [&](float2 vh, float2 vl, float2& nSh, float2& Sl) {
            const float2 np = __fmul2_rn(vh, nc3);  // -(v c3), whose error the fma below gives
            float2 e = __ffma2_rn(vh, c3, np);
            e = __ffma2_rn(vh, cl, e);
            e = __ffma2_rn(vl, c3, e);
            float2 u;
            two_sum2(nSh, np, nSh, u);
            Sl = __fadd2_rn(Sl, __ffma2_rn(u, m1, e));
        };
        add(xh, xl, S.xh, S.xl);
        add(yh, yl, S.yh, S.yl);
        add(zh, zl, S.zh, S.zl);
    }
    // degrees 2 to 4 in FP32
    const float2 s = __fmul2_rn(y0, bc2(rho)), s2 = __fmul2_rn(s, s);
    const float2 nx = __fmul2_rn(xh, y0), nz = __fmul2_rn(zh, y0);
    const float2 qxx = __fmul2_rn(nx, nx), qxz = __fmul2_rn(nx, nz), qzz = __fmul2_rn(nz, nz);
    const float2 qd = __fadd2_rn(qxz, qxz);
    const float4 m0 = mom[0], m1_ = mom[1];
    const float2 w2x = __ffma2_rn(lane2(m0, 0), nx, __fmul2_rn(lane2(m0, 1), nz));
    const float2 w2z = __ffma2_rn(lane2(m0, 1), nx, __fmul2_rn(lane2(m1_, 0), nz));
    const float2 T2 = __ffma2_rn(w2x, nx, __fmul2_rn(w2z, nz));
    const float4 m2 = mom[2], m3 = mom[3], m4 = mom[4];
    const float2 ntx = lane2(m4, 0), ntz = lane2(m4, 1);
    const float2 w3x =
        __ffma2_rn(lane2(m2, 0), qxx, __ffma2_rn(lane2(m2, 1), qd, __ffma2_rn(lane2(m3, 0), qzz, ntx)));
    const float2 w3z =
        __ffma2_rn(lane2(m2, 1), qxx, __ffma2_rn(lane2(m3, 0), qd, __ffma2_rn(lane2(m3, 1), qzz, ntz)));
    const float2 W3 = __ffma2_rn(w3x, nx, __fmul2_rn(w3z, nz));
    const float2 ntn = __ffma2_rn(ntx, nx, __fmul2_rn(ntz, nz));
    const float4 m5 = mom[5], m6 = mom[6], m7 = mom[7], m8 = mom[8], m9 = mom[9], m10 = mom[10];
    const float2 T22 = lane2(m7, 1), P20 = lane2(m8, 1), P11 = lane2(m9, 0), P02 = lane2(m9, 1);
    const float2 gx =
        __ffma2_rn(lane2(m5, 0), qxx, __ffma2_rn(lane2(m7, 0), qxz, __ffma2_rn(T22, qzz, P20)));
    const float2 gz =
        __ffma2_rn(lane2(m6, 1), qzz, __ffma2_rn(lane2(m8, 0), qxz, __ffma2_rn(T22, qxx, P02)));
    const float2 w4x = __ffma2_rn(nx, gx, __fmul2_rn(nz, __ffma2_rn(lane2(m6, 0), qzz, P11)));
    const float2 w4z = __ffma2_rn(nz, gz, __fmul2_rn(nx, __ffma2_rn(lane2(m5, 1), qxx, P11)));
    const float2 W4 = __ffma2_rn(w4x, nx, __fmul2_rn(w4z, nz));
    const float2 Q = __ffma2_rn(P20, qxx, __ffma2_rn(P11, qd, __fmul2_rn(P02, qzz)));
    if constexpr (kPhi) {
        const float2 f2 = __ffma2_rn(bc2(0.5f), T2, lane2(m1_, 1));
        const float2 f3 = __ffma2_rn(bc2(1.f / 3.f), W3, __fmul2_rn(bc2(2.f / 3.f), ntn));
        const float2 f4 = __ffma2_rn(bc2(0.25f), __fadd2_rn(W4, Q), lane2(m10, 0));
        const float2 f = __ffma2_rn(s2, f4, __ffma2_rn(s, f3, f2));
        S.fc = __ffma2_rn(c3, f, S.fc);
    }
    if constexpr (kField) {
        const float2 ny = __fmul2_rn(yh, y0);
        const float2 r2 = __ffma2_rn(bc2(2.5f), T2, lane2(mom[11], 0));
        const float2 r3 = __ffma2_rn(bc2(7.f / 3.f), W3, __fmul2_rn(bc2(8.f / 3.f), ntn));
        const float2 r4 = __ffma2_rn(bc2(2.25f), W4, __ffma2_rn(bc2(1.25f), Q, lane2(m10, 1)));
        const float2 r = __ffma2_rn(s2, r4, __ffma2_rn(s, r3, r2));
        const float2 wx = __ffma2_rn(s2, w4x, __ffma2_rn(s, w3x, w2x));
        const float2 wz = __ffma2_rn(s2, w4z, __ffma2_rn(s, w3z, w2z));
        const float2 k = __fmul2_rn(c3, s), nk = __fmul2_rn(k, m1), kr = __fmul2_rn(k, r);
        S.ex = __ffma2_rn(nk, wx, __ffma2_rn(kr, nx, S.ex));
        S.ey = __ffma2_rn(kr, ny, S.ey);
        S.ez = __ffma2_rn(nk, wz, __ffma2_rn(kr, nz, S.ez));
    }
}

}  // namespace nb
