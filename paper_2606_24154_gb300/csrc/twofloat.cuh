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
    // (distances beyond 1e-19 m: normal numbers)
    y0 = make_float2(rsqrt_normal(r2h.x), rsqrt_normal(r2h.y));
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
    const float2 y0 = make_float2(far0 ? rsqrt_normal(d2h.x) : 0.f, far1 ? rsqrt_normal(d2h.y) : 0.f);
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

// ---------------------------------------------------------------- far pairs of the fill by moments
// Phi' or n . E' of a pair from kFillRatioB = 32 radii on, to the fill's accuracy, two images per packed
// instruction.  With y = 1 / |D|, p = y^2, N = n . D and all moments over the area A:
//   Phi' / A   = y (1 + W + F),  W = q p Q,  Q = a1 X^2 + a2 X Z + a3 Z^2 - w |D|^2 (degree 2),
//   n . E' / A = y p (N (1 + 5 W + G) - q H - s (n_x F_alpha + n_z F_beta)),  H = n . grad Q,
//   F(alpha, beta, q) = terms of degree 3 to 6,  alpha = X p s, beta = Z p s, q = p s^2,
//   G = F + 2 (alpha F_alpha + beta F_beta + q F_q).
// s = the power of two above the element's radius: the moments, of (node - centroid) / s, stay FP32 numbers
// at any size of the geometry, and q is exact.
// The monopole and the quadrupole (below 1.5e-4 of the pair) are in two-float arithmetic, F (below
// 1.5e-6) in FP32; the terms left out (degree 7) are below 3e-13 at 32 radii.  In the field they count
// eight times as much, so interface rows use the moments from kFillMomField = 52 radii on.  150 (Phi') and
// 376 (n . E') FP32 lane operations after the pair's geometry (51) and one MUFU root per pair, where the
// 6, 9 and 16 nodes of the Gauss rules took 390 to 920 and 640 to 1540 and as many roots.
// FillMom per element, every constant twice (both lanes), two per float4: a1, a2, a3, -w as hi, lo, then
// the coefficients of F in the order of fill_mom_off, then A as hi, lo, s, s^2.
constexpr double kFillMomField = 52.0;
constexpr int kFillMomCoef = 43;
constexpr int kFillMomF4 = (8 + kFillMomCoef + 1) / 2 + 1;
// F's monomials alpha^i beta^j, i + j = k <= 6: coefficient q^m0 (C + C' q), m0 and the number of terms
__host__ __device__ constexpr int fill_mom_m0(int k) { return k == 0 ? 2 : k <= 2 ? 1 : 0; }
__host__ __device__ constexpr int fill_mom_terms(int k) { return k <= 4 ? 2 : 1; }
__host__ __device__ constexpr int fill_mom_off(int i, int j) {
    int o = 0;
    for (int b = 0; b < 7; ++b)
        for (int a = 0; a + b < 7; ++a) {
            if (a == i && b == j) return o;
            o += fill_mom_terms(a + b);
        }
    return o;
}
static_assert(fill_mom_off(0, 6) + 1 == kFillMomCoef, "coefficient count");

// (vh, vl) = (ah, al) (vh, vl)
__device__ __forceinline__ void df_times2(float2 ah, float2 al, float2& vh, float2& vl) {
    const float2 t = __fmul2_rn(ah, vh);
    const float2 e = __ffma2_rn(ah, vh, __fmul2_rn(t, bc2(-1.f)));
    vl = __ffma2_rn(ah, vl, __ffma2_rn(al, vh, e));
    vh = t;
}

// Two targets (lanes) of an element: X, Z and |D|^2 with the squares that it was summed from.
struct FillPair2 {
    float2 xh, xl, zh, zl, px, ex, pz, ez, d2h, d2l;
};
// A conductor row's sum; the interface row's takes the normal and H's constants in the element's frame.
struct FillRow {
    float nxh, nxl, nyh, nyl, nzh, nzl;  // n in the element's frame
    float gxh, gxl, gzh, gzl;            // 2 a1 n_x + a2 n_z, a2 n_x + 2 a3 n_z
};

// 1 / |D| of the lanes that are far (0 of the others) as y0 + ye, its square p as a + al, q and W
__device__ __forceinline__ void fill_mom_head2(const float4* __restrict__ mom, const FillPair2& P, bool far0, bool far1,
                                               float2& y0, float2& ye, float2& a, float2& al, float2& q, float2& ql, float2& W,
                                               float2& lo) {
    const float2 m1 = bc2(-1.f);
    auto con = [&](int i) { return lane2(mom[i >> 1], i & 1); };
    y0 = make_float2(far0 ? rsqrt_normal(P.d2h.x) : 0.f, far1 ? rsqrt_normal(P.d2h.y) : 0.f);
    const float2 ny0 = __fmul2_rn(y0, m1);
    a = __fmul2_rn(y0, y0);
    const float2 na = __fmul2_rn(ny0, y0);
    const float2 nae = __ffma2_rn(ny0, y0, a);  // a - y0^2
    const float2 b = __fmul2_rn(P.d2h, a);
    const float2 nbe = __ffma2_rn(P.d2h, na, b);
    float2 h = __ffma2_rn(b, m1, bc2(1.f));
    h = __fadd2_rn(h, nbe);
    h = __ffma2_rn(P.d2h, nae, h);
    h = __ffma2_rn(P.d2l, na, h);
    ye = __fmul2_rn(__fmul2_rn(bc2(0.5f), y0), h);
    al = __ffma2_rn(nae, m1, __fmul2_rn(__fadd2_rn(y0, y0), ye));
    // Q: four products of two-float numbers, summed with their errors
    const float2 pxz = __fmul2_rn(P.xh, P.zh);
    float2 exz = __ffma2_rn(P.xh, P.zh, __fmul2_rn(pxz, m1));
    exz = __ffma2_rn(P.xh, P.zl, __ffma2_rn(P.xl, P.zh, exz));
    lo = bc2(0.f);
    auto product = [&](int i, float2 vh, float2 vl) {
        const float2 ch = con(2 * i), cl = con(2 * i + 1);
        const float2 t = __fmul2_rn(ch, vh);
        lo = __fadd2_rn(lo, __ffma2_rn(ch, vh, __fmul2_rn(t, m1)));
        lo = __ffma2_rn(ch, vl, __ffma2_rn(cl, vh, lo));
        return t;
    };
    const float2 t1 = product(0, P.px, P.ex), t2 = product(1, pxz, exz), t3 = product(2, P.pz, P.ez),
                 t4 = product(3, P.d2h, P.d2l);
    float2 e1, e2, e3;
    two_sum2(t1, t3, W, e1);
    two_sum2(W, t2, W, e2);
    two_sum2(W, t4, W, e3);
    lo = __fadd2_rn(lo, __fadd2_rn(e1, __fadd2_rn(e2, e3)));
    const float2 ss = bc2(mom[kFillMomF4 - 1].w);
    q = __fmul2_rn(a, ss), ql = __fmul2_rn(al, ss);
    df_times2(a, al, W, lo);
    df_times2(q, ql, W, lo);
}

// (Sh, Sl) += y (1 + W + F) of the lanes that are far
__device__ __forceinline__ void fill_mom_phi2(const float4* __restrict__ mom, const FillPair2& P, bool far0,
                                              bool far1, float2& Sh, float2& Sl) {
    auto con = [&](int i) { return lane2(mom[i >> 1], i & 1); };
    float2 y0, ye, a, al, q, ql, W, lo;
    fill_mom_head2(mom, P, far0, far1, y0, ye, a, al, q, ql, W, lo);
    df_times2(y0, ye, W, lo);
    const float2 pr = __fmul2_rn(a, bc2(mom[kFillMomF4 - 1].z)), qq = __fmul2_rn(q, q);
    const float2 al1 = __fmul2_rn(P.xh, pr), be1 = __fmul2_rn(P.zh, pr);
    float2 F = bc2(0.f);
#pragma unroll
    for (int j = 6; j >= 0; --j) {
        float2 R = bc2(0.f);
#pragma unroll
        for (int i = 6 - j; i >= 0; --i) {
            const int o = 8 + fill_mom_off(i, j), k = i + j;
            float2 c = con(o);
            if (fill_mom_terms(k) == 2) c = __ffma2_rn(con(o + 1), q, c);
            if (fill_mom_m0(k) == 1) c = __fmul2_rn(c, q);
            if (fill_mom_m0(k) == 2) c = __fmul2_rn(c, qq);
            R = i == 6 - j ? c : __ffma2_rn(R, al1, c);
        }
        F = j == 6 ? R : __ffma2_rn(F, be1, R);
    }
    float2 u1, u2;
    two_sum2(Sh, y0, Sh, u1);
    two_sum2(Sh, W, Sh, u2);
    lo = __fadd2_rn(lo, __fadd2_rn(ye, __fadd2_rn(u1, u2)));
    Sl = __fadd2_rn(Sl, __ffma2_rn(y0, F, lo));
}

// F, G, F_alpha, F_beta by Horner's rule (qq = q^2)
__device__ __forceinline__ void fill_mom_poly2(const float4* __restrict__ mom, float2 al1, float2 be1, float2 q,
                                               float2 qq, float2& F, float2& G, float2& Fa, float2& Fb) {
    auto con = [&](int i) { return lane2(mom[i >> 1], i & 1); };
    F = G = Fa = Fb = bc2(0.f);
#pragma unroll
    for (int j = 6; j >= 0; --j) {
        float2 r = bc2(0.f), ra = bc2(0.f), rg = bc2(0.f);
#pragma unroll
        for (int i = 6 - j; i >= 0; --i) {
            const int o = 8 + fill_mom_off(i, j), k = i + j;
            const float f0 = (float)(1 + 2 * (k + fill_mom_m0(k)));
            float2 c = con(o), g;
            if (fill_mom_terms(k) == 2) {
                const float2 c1 = __fmul2_rn(con(o + 1), q);
                c = __fadd2_rn(c, c1);
                g = __ffma2_rn(c1, bc2(2.f), __fmul2_rn(c, bc2(f0)));
            } else {
                g = __fmul2_rn(c, bc2(f0));
            }
            if (fill_mom_m0(k) == 1) c = __fmul2_rn(c, q), g = __fmul2_rn(g, q);
            if (fill_mom_m0(k) == 2) c = __fmul2_rn(c, qq), g = __fmul2_rn(g, qq);
            if (i == 6 - j) {
                r = c, rg = g;
            } else {
                ra = i == 5 - j ? r : __ffma2_rn(ra, al1, r);
                r = __ffma2_rn(r, al1, c);
                rg = __ffma2_rn(rg, al1, g);
            }
        }
        if (j == 6) {
            F = r, G = rg;
        } else {
            Fb = j == 5 ? F : __ffma2_rn(Fb, be1, F);
            F = __ffma2_rn(F, be1, r);
            G = __ffma2_rn(G, be1, rg);
            Fa = j == 5 ? ra : __ffma2_rn(Fa, be1, ra);
        }
    }
}

// (Sh, Sl) += n . E' / A of the lanes that are far; (yh, yl) = the targets' Y
__device__ __forceinline__ void fill_mom_field2(const float4* __restrict__ mom, const FillRow& R,
                                                const FillPair2& P, float2 yh, float2 yl, bool far0, bool far1,
                                                float2& Sh, float2& Sl) {
    const float2 m1 = bc2(-1.f);
    auto con = [&](int i) { return lane2(mom[i >> 1], i & 1); };
    auto product = [&](float ch, float cl, float2 vh, float2 vl, float2& e) {  // its hi; e += its lo
        const float2 t = __fmul2_rn(bc2(ch), vh);
        e = __fadd2_rn(e, __ffma2_rn(bc2(ch), vh, __fmul2_rn(t, m1)));
        e = __ffma2_rn(bc2(ch), vl, __ffma2_rn(bc2(cl), vh, e));
        return t;
    };
    float2 y0, ye, a, al, q, ql, W, wl;
    fill_mom_head2(mom, P, far0, far1, y0, ye, a, al, q, ql, W, wl);
    float2 Nh, Nl = bc2(0.f), e1, e2;
    const float2 n1 = product(R.nxh, R.nxl, P.xh, P.xl, Nl), n2 = product(R.nyh, R.nyl, yh, yl, Nl),
                 n3 = product(R.nzh, R.nzl, P.zh, P.zl, Nl);
    two_sum2(n1, n2, Nh, e1);
    two_sum2(Nh, n3, Nh, e2);
    Nl = __fadd2_rn(Nl, __fadd2_rn(e1, e2));
    // q H, H = gx X + gz Z - 2 w N
    float2 Hh, Hl = bc2(0.f);
    const float2 h1 = product(R.gxh, R.gxl, P.xh, P.xl, Hl), h2 = product(R.gzh, R.gzl, P.zh, P.zl, Hl);
    float2 h3 = __fadd2_rn(con(6), con(6)), h3l = __fadd2_rn(con(7), con(7));  // -2 w
    {
        float2 vh = Nh, vl = Nl;
        df_times2(h3, h3l, vh, vl);
        h3 = vh;
        Hl = __fadd2_rn(Hl, vl);
    }
    two_sum2(h1, h2, Hh, e1);
    two_sum2(Hh, h3, Hh, e2);
    Hl = __fadd2_rn(Hl, __fadd2_rn(e1, e2));
    df_times2(q, ql, Hh, Hl);
    // 5 W N
    df_times2(bc2(5.f), bc2(0.f), W, wl);
    df_times2(Nh, Nl, W, wl);
    // G, F_alpha, F_beta
    const float s = mom[kFillMomF4 - 1].z;
    const float2 pr = __fmul2_rn(a, bc2(s)), qq = __fmul2_rn(q, q);
    const float2 al1 = __fmul2_rn(P.xh, pr), be1 = __fmul2_rn(P.zh, pr);
    float2 F, G, Fa, Fb;
    fill_mom_poly2(mom, al1, be1, q, qq, F, G, Fa, Fb);
    // T = N + 5 W N - q H + FP32 part, then y p T
    float2 Th, Tl;
    two_sum2(Nh, W, Th, e1);
    two_sum2(Th, __fmul2_rn(Hh, m1), Th, e2);
    Tl = __fadd2_rn(__fadd2_rn(Nl, wl), __fadd2_rn(e1, e2));
    Tl = __ffma2_rn(Hl, m1, Tl);
    const float2 D = __ffma2_rn(bc2(R.nxh), Fa, __fmul2_rn(bc2(R.nzh), Fb));
    Tl = __fadd2_rn(Tl, __ffma2_rn(Nh, G, __fmul2_rn(D, bc2(-s))));
    df_times2(a, al, Th, Tl);
    df_times2(y0, ye, Th, Tl);
    float2 u;
    two_sum2(Sh, Th, Sh, u);
    Sl = __fadd2_rn(Sl, __fadd2_rn(u, Tl));
}

// Sums of fill_mom_point2: phi / A and E (local frame) / A, both lanes, two floats each.
struct PointSum2 {
    float2 ph, pl, xh, xl, yh, yl, zh, zl;
};
// S += Phi' / A and E' / A (the vector) of the lanes that are far: as fill_mom_phi2, and with
// T = 5 W + 2 q w + G
//   E'_x / A = y p (X (1 + T) - q (2 a1 X + a2 Z) - s F_alpha),   E'_y / A = y p Y (1 + T),
// E'_z like E'_x.  About 400 FP32 lane operations.
__device__ __forceinline__ void fill_mom_point2(const float4* __restrict__ mom, const FillPair2& P, float2 yh, float2 yl,
                                                bool far0, bool far1, PointSum2& S) {
    const float2 m1 = bc2(-1.f);
    auto con = [&](int i) { return lane2(mom[i >> 1], i & 1); };
    float2 y0, ye, a, al, q, ql, W, wl;
    fill_mom_head2(mom, P, far0, far1, y0, ye, a, al, q, ql, W, wl);
    // F, G, F_alpha, F_beta
    const float s = mom[kFillMomF4 - 1].z;
    const float2 pr = __fmul2_rn(a, bc2(s)), qq = __fmul2_rn(q, q);
    const float2 al1 = __fmul2_rn(P.xh, pr), be1 = __fmul2_rn(P.zh, pr);
    float2 F, G, Fa, Fb;
    fill_mom_poly2(mom, al1, be1, q, qq, F, G, Fa, Fb);
    float2 t, u;
    {  // y (1 + W + F)
        float2 vh = W, vl = wl;
        df_times2(y0, ye, vh, vl);
        two_sum2(S.ph, y0, S.ph, t);
        two_sum2(S.ph, vh, S.ph, u);
        vl = __fadd2_rn(vl, __fadd2_rn(ye, __fadd2_rn(t, u)));
        S.pl = __fadd2_rn(S.pl, __ffma2_rn(y0, F, vl));
    }
    // T
    float2 ch = q, cl = ql, Th, Tl;
    df_times2(__fmul2_rn(con(6), bc2(-2.f)), __fmul2_rn(con(7), bc2(-2.f)), ch, cl);
    df_times2(bc2(5.f), bc2(0.f), W, wl);
    two_sum2(W, ch, Th, t);
    Tl = __fadd2_rn(__fadd2_rn(wl, cl), __fadd2_rn(t, G));
    df_times2(y0, ye, a, al);  // y p
    // component: (c (1 + T) - q g - s f) y p, g = gx X + gz Z (0 without in_plane)
    auto component = [&](float2 h, float2 l, bool in_plane, int ix, float fx, int iz, float fz, float2 f, float2& Sh,
                         float2& Sl) {
        float2 vh = Th, vl = Tl, rh, e, g;
        df_times2(h, l, vh, vl);
        two_sum2(h, vh, rh, e);
        vl = __fadd2_rn(__fadd2_rn(l, vl), e);
        if (in_plane) {
            float2 gh = __fmul2_rn(con(ix), bc2(fx)), gl = __fmul2_rn(con(ix + 1), bc2(fx));
            float2 kh = __fmul2_rn(con(iz), bc2(fz)), kl = __fmul2_rn(con(iz + 1), bc2(fz));
            df_times2(P.xh, P.xl, gh, gl);
            df_times2(P.zh, P.zl, kh, kl);
            two_sum2(gh, kh, g, e);
            gl = __fadd2_rn(__fadd2_rn(gl, kl), e);
            df_times2(q, ql, g, gl);
            two_sum2(rh, __fmul2_rn(g, m1), rh, e);
            vl = __fadd2_rn(__ffma2_rn(gl, m1, vl), __ffma2_rn(f, bc2(-s), e));
        }
        df_times2(a, al, rh, vl);
        two_sum2(Sh, rh, Sh, e);
        Sl = __fadd2_rn(Sl, __fadd2_rn(vl, e));
    };
    component(P.xh, P.xl, true, 0, 2.f, 2, 1.f, Fa, S.xh, S.xl);
    component(yh, yl, false, 0, 0.f, 0, 0.f, Fa, S.yh, S.yl);
    component(P.zh, P.zl, true, 2, 1.f, 4, 2.f, Fb, S.zh, S.zl);
}

}  // namespace nb
