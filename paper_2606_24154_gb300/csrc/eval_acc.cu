// eval_acc.cu -- refinement of the mixed-precision evaluation (Eq. Potential / Eq. Field
// over elements and periodic images): per-point error estimates of the FP32 pass, and a
// two-float re-evaluation of the points whose estimate exceeds the requested tolerance.
//
// Error estimate.  The FP32 pass (eval_blocks.cuh) leaves per point the scales of its FP32
// pairs' errors, built from the per-element terms b_j = |sigma_j| |sum_k Phi'_jk| (for E:
// |sigma_j| |sum_k E'_jk|_1): B = ke sum_j b_j and S = ke sqrt(sum_j b_j^2).  Its error
// comes from rounding the point-to-centroid difference and the node arithmetic to FP32
// (about u = 2^-24 relative per operation) and from the truncation of the Gauss rules.
// These do not shrink with the result, so a point whose |phi| (|E|) is small next to B --
// a potential near zero inside the plate, the weak field in the drift gap -- loses its
// relative accuracy there.  The estimate for x = phi and x = |E| is
//   gamma_r |x| + gamma_b B + gamma_s S,   gamma_r = 1e-7, gamma_b = 7e-8, gamma_s = 5e-7.
// Calibration: against the FP64 path on 133,000 points (the THGEM cell with solved and
// with structured densities, points in the gas, through the plate and 1-2 um off the Cu
// faces; the cube with solved densities on its grid and at random points; a reduced THGEM
// cell), the largest error ratios were 3.3e-8 B (phi) and 5.5e-8 B (E) on the THGEM cell
// and 7.7e-8 of the result on the cube and the reduced cell, where B and the result are
// close.  The constants cover every one of those errors by 1.7x or more (2x for phi).
// Most of the error follows B, not S: many pairs round alike (every element of a plane sees
// a point at the same z offset, identical elements carry identical FP32 node tables), so
// their errors keep one sign instead of averaging out; the S term covers the rest.  The
// estimate is statistical, not a bound.  The constants can be changed per context
// (nebem_set_error_model).
//
// Refinement.  A point is re-evaluated when its estimate exceeds tol |phi| or tol |E|,
// in two-float arithmetic (about 44 bits; the error-free transformations of twofloat.cuh),
// in two levels.  Level 1 takes the pairs from 28 radii on by the element's moments (two-float
// monopole, degrees 2 to 4 in FP32) and the nearer ones by the FP32 pass's Gauss rules and FP64 near
// pairs: its error, measured against the closed forms on THGEM points, stays below
// ~2e-11 of B; its estimate is 1e-9 B.  Points whose level-1 estimate still exceeds the
// tolerance go to level 2, the arithmetic of the mixed fill (fill_mixed.cu: moments with a two-float
// quadrupole from 40 radii on, rules truncated below ~3e-12 of each pair nearer, FP64 closed forms
// within kFillRatioC element radii), estimate 1e-11 B.  In the frame of element j (axes ex, ey = normal,
// ez), a pair (point, image k) has D = P - c_j - t_k with local components X = (P - c_j) . ex - tau_k.x
// (likewise Y, Z; tau tabulated per element and image), from which the moments' series follow
// (twofloat.cuh); a node at offset s = centroid - node (in the element plane) sees the point at D + s, so r^2 = |D|^2 + 2 (X s_x + Z s_z) + |s|^2 and
//   Phi' = sum w / r,   E'_local = D sum w / r^3 + (sum w s_x / r^3, 0, sum w s_z / r^3).
// Per element the image sums are rotated to the global frame and weighted by sigma_j in
// FP64.  Every flagged point's arithmetic depends on that point only, so its result does
// not depend on which other points are flagged or share the launch.
#include "twofloat.cuh"

namespace nb {

namespace {

constexpr int kAT = 128;             // threads (flagged points) per block
constexpr int kATBlocks = 5;         // resident far blocks per SM (96 registers a thread)
constexpr double kErrGammaR = 1e-7;   // FP32 pass: share of the result
constexpr double kErrGammaB = 7e-8;   // FP32 pass: share of B
constexpr double kErrGammaS = 5e-7;   // FP32 pass: share of S
constexpr double kGammaL1 = 1e-9;    // two-float, the FP32 pass's rules (truncation ~1e-10 B)
constexpr double kGammaL2 = 1e-11;   // two-float, fill-grade rules
constexpr double kMomRatio2 = 40.0;  // level 2: the radius from which the fill's moments are taken (truncation 5e-13 of E)

// What a refinement pass re-evaluates: both phi and E, phi only (its E estimate was within
// the tolerance, E keeps the FP32 pass's value), or E only.
constexpr int kBoth = 0, kPhiOnly = 1, kEOnly = 2;

// Per-pair node sums S0 = sum w / r^3, S2x = sum w (2 s_x) / r^3, S2z = sum w (2 s_z) / r^3
// as packed two-float values (hi, negated lo) over the two lanes of the node pairs.
struct PairSums2 {
    float2 s0, ns0, sx, nsx, sz, nsz;
};

// Phi' (per element, accumulated over its images: ph, nph) and the pair sums of one tier's
// node pairs.  Node records as in nb_internal.h (kFillNodeRec layout): q0 = (2 s_x, 2 s_z)
// hi, q1 = (|s|^2, w) hi, q2 / q3 the lo parts.
template <int M>
__device__ __forceinline__ void nodes_acc2(const float4* __restrict__ nd, int pairs, const PairDF2& P, float2& ph,
                                           float2& nph, PairSums2& S) {
    const float2 m1 = bc2(-1.f);
    for (int q = 0; q < pairs; ++q) {
        const float4 q0 = nd[4 * q], q1 = nd[4 * q + 1], q2 = nd[4 * q + 2], q3 = nd[4 * q + 3];
        float2 y0, ny0, nyl, a, na, nae;
        node_rinv2(P, q0, q1, q2, q3, y0, ny0, nyl, a, na, nae);
        const float2 w = make_float2(q1.z, q1.w), wl = make_float2(q3.z, q3.w);
        float2 t;
        if constexpr (M != kEOnly) {
            // w / r = m - nme
            const float2 m = __fmul2_rn(w, y0);
            float2 nme = __ffma2_rn(w, ny0, m);
            nme = __ffma2_rn(w, nyl, nme);
            nme = __ffma2_rn(wl, ny0, nme);
            two_sum2(ph, m, ph, t);
            nph = __ffma2_rn(t, m1, __fadd2_rn(nph, nme));
        }
        if constexpr (M == kPhiOnly) continue;
        // y^3 = c3 - nc3e (y^2 = a - ny2l)
        const float2 ny2l = __ffma2_rn(__fadd2_rn(y0, y0), nyl, nae);
        const float2 c3 = __fmul2_rn(a, y0);
        float2 nc3e = __ffma2_rn(na, y0, c3);
        nc3e = __ffma2_rn(a, nyl, nc3e);
        nc3e = __ffma2_rn(ny2l, y0, nc3e);
        const float2 nc3 = __fmul2_rn(c3, m1);
        // w y^3 = m3 - nm3e
        const float2 m3 = __fmul2_rn(w, c3);
        float2 nm3e = __ffma2_rn(w, nc3, m3);
        nm3e = __ffma2_rn(w, nc3e, nm3e);
        nm3e = __ffma2_rn(wl, nc3, nm3e);
        two_sum2(S.s0, m3, S.s0, t);
        S.ns0 = __ffma2_rn(t, m1, __fadd2_rn(S.ns0, nm3e));
        // (w y^3) (2 s_x), (w y^3) (2 s_z)
        const float2 nm3 = __fmul2_rn(m3, m1);
        const float2 sx = make_float2(q0.x, q0.y), sz = make_float2(q0.z, q0.w);
        const float2 sxl = make_float2(q2.x, q2.y), szl = make_float2(q2.z, q2.w);
        const float2 fx = __fmul2_rn(m3, sx);
        float2 nfx = __ffma2_rn(nm3, sx, fx);
        nfx = __ffma2_rn(nm3, sxl, nfx);
        nfx = __ffma2_rn(nm3e, sx, nfx);
        two_sum2(S.sx, fx, S.sx, t);
        S.nsx = __ffma2_rn(t, m1, __fadd2_rn(S.nsx, nfx));
        const float2 fz = __fmul2_rn(m3, sz);
        float2 nfz = __ffma2_rn(nm3, sz, fz);
        nfz = __ffma2_rn(nm3, szl, nfz);
        nfz = __ffma2_rn(nm3e, sz, nfz);
        two_sum2(S.sz, fz, S.sz, t);
        S.nsz = __ffma2_rn(t, m1, __fadd2_rn(S.nsz, nfz));
    }
}

// the two lanes of a packed (hi, negated lo) sum as one two-float value, times `scale`
// (a power of two, exact)
__device__ __forceinline__ void lanes_to_df(float2 h, float2 nl, float scale, float& oh, float& ol) {
    float t;
    two_sum(h.x, h.y, oh, t);
    ol = __fsub_rn(__fsub_rn(t, nl.x), nl.y);
    oh = __fmul_rn(oh, scale);
    ol = __fmul_rn(ol, scale);
}

// (Sh, Sl) += (ah + al) (bh + bl) + (ch + cl)
__device__ __forceinline__ void df_fma_acc(float ah, float al, float bh, float bl, float ch, float cl, float& Sh,
                                           float& Sl) {
    const float p = __fmul_rn(ah, bh);
    float e = __fmaf_rn(ah, bh, -p);
    e = __fmaf_rn(ah, bl, e);
    e = __fmaf_rn(al, bh, e);
    float h, t, t2;
    two_sum(p, ch, h, t);
    const float l = __fadd_rn(e, __fadd_rn(t, cl));
    two_sum(Sh, h, Sh, t2);
    Sl = __fadd_rn(Sl, __fadd_rn(t2, l));
}

// Two levels of re-evaluation, both two-float: level 1 takes the pairs from kMomRatio radii on by
// their moments (mom_pair2) and the nearer ones by the tiers of the FP32 pass (nb_internal.h
// FarNodes: 3x3 / 6-point, 4x4, 6x6 rules at ratio_a, ratio_b, ratio_near radii; FP64 closed forms
// nearer); its truncation stays near 1e-10 of B.  Level 2 takes the pairs from kMomRatio2 radii
// on by the fill's moments (fill_mom_point2) and the nearer ones by the fill's tiers (truncation
// below ~3e-12 of each pair, FP64 within kFillRatioC radii).
//
// dynamic shared memory per tile of te elements: FillEl (9 float4), the level's moments, the tier
// radii, and tau as six planes of nimg (padded to even) floats (x, y, z negated: hi, then lo).
__host__ __device__ constexpr int acc_pad(int nimg) { return (nimg + 1) & ~1; }
// odd strides (moments in float4, tau in float2): the lanes of the lane path read different elements
__host__ __device__ constexpr int acc_tau_stride(int nimg) { return 6 * acc_pad(nimg) + 2; }
__host__ __device__ constexpr int acc_mom_f4(int level) { return (level == 1 ? kMomF4 : kFillMomF4) | 1; }
__host__ __device__ constexpr int acc_tile_f4(int level, int te, int nimg) {
    return te * (9 + acc_mom_f4(level) + 1) + (te * acc_tau_stride(nimg) + 3) / 4;
}

// A unit of the lane path (acc_range): kLP points of one leaf.  Per warp the values (sigma, Phi', E') of 32
// (point, element) pairs, and the chains' results (Sum6) of its points.
constexpr int kLP = 8;
// Lists whose units are few take the lane path.  A thread per point cannot end before one thread has taken
// its leaf, however short the list (0.9 ms at level 1 and 2.4 ms at level 2 for 10,000 elements x 25 copies);
// with the lane path 20 points take 0.11 and 0.32 ms, 257 take 0.84 and 2.5 (1.7 and 4.0), 500 1.5 and
// 4.0 (2.1 and 4.9), and from about 1,000 points (50 units per resident block) on both are alike.
constexpr int64_t kLaneRounds = 32;
__host__ __device__ __forceinline__ bool lane_path(const SplitPlan& plan, int64_t count, int64_t gb) {
    return plan.leaf && plan.Gm == 0 && (count + kLP - 1) / kLP * plan.np < kLaneRounds * gb;
}
struct LaneScratch {
    struct Val {  // d: sigma, Phi', E'; for the scales a: |Phi'|, |E'|_1
        double d[5], a[2];
    };
    Val val[kAT / 32][32];
    double out[kLP][6];
};

// Sums of an element's nearer pairs (those not taken by moments), two floats each.
struct NearerSum {
    float ph, pl, xh, xl, yh, yl, zh, zl;
};

// One such pair by its tier's nodes: Phi' and E' (local) added to N.  About one pair in a hundred; kept
// out of line and out of the image loop, whose registers it would otherwise crowd.
template <int M>
__device__ __noinline__ void acc_pair_nodes(const AccView& A, const float4& hdr, int na, int64_t j, int nimg, int k,
                                            const float (&ph)[3], const float (&pl)[3], float x0h, float x0l, float y0h,
                                            float y0l, float z0h, float z0l, const float* __restrict__ tau, int np2,
                                            NearerSum& N) {
    const int64_t jk = j * nimg + k;
    float dx, dy, dz;
    const float d2 = pair_d2(ph[0], ph[1], ph[2], pl[0], pl[1], pl[2], A.cjk[2 * jk], A.cjk[2 * jk + 1], dx, dy, dz);
    if (!(d2 >= hdr.w)) return;  // near pair: the FP64 kernel
    const float4* nd = A.nodes + j * kFillNodeRec;
    int np = na;
    if (!(d2 >= hdr.y)) {
        const bool b = d2 >= hdr.z;
        nd += b ? kFillOffB : kFillOffC;
        np = b ? kFillPairsB : kFillPairsC;
    }
    float xh, xl, yh, yl, zh, zl, d2h, d2l;
    df_sub(x0h, x0l, -tau[k], -tau[3 * np2 + k], xh, xl);
    df_sub(y0h, y0l, -tau[np2 + k], -tau[4 * np2 + k], yh, yl);
    df_sub(z0h, z0l, -tau[2 * np2 + k], -tau[5 * np2 + k], zh, zl);
    df_norm2(xh, xl, yh, yl, zh, zl, d2h, d2l);
    PairDF2 P;
    P.xh = bc2(xh), P.nxh = bc2(-xh), P.xl = bc2(xl);
    P.zh = bc2(zh), P.nzh = bc2(-zh), P.zl = bc2(zl);
    P.d2h = bc2(d2h), P.d2l = bc2(d2l);
    PairSums2 S{bc2(0.f), bc2(0.f), bc2(0.f), bc2(0.f), bc2(0.f), bc2(0.f)};
    float2 sh = bc2(0.f), snl = bc2(0.f);
    nodes_acc2<M>(nd, np, P, sh, snl, S);
    if constexpr (M != kEOnly) {
        float h, l, t;
        lanes_to_df(sh, snl, 1.f, h, l);
        two_sum(N.ph, h, N.ph, t);
        N.pl = __fadd_rn(N.pl, __fadd_rn(t, l));
    }
    if constexpr (M != kPhiOnly) {
        float s0h, s0l, sxh, sxl, szh, szl;
        lanes_to_df(S.s0, S.ns0, 1.f, s0h, s0l);
        lanes_to_df(S.sx, S.nsx, 0.5f, sxh, sxl);
        lanes_to_df(S.sz, S.nsz, 0.5f, szh, szl);
        df_fma_acc(xh, xl, s0h, s0l, sxh, sxl, N.xh, N.xl);
        df_fma_acc(yh, yl, s0h, s0l, 0.f, 0.f, N.yh, N.yl);
        df_fma_acc(zh, zl, s0h, s0l, szh, szl, N.zh, N.zl);
    }
}

// Level 1, 1e6 points of the 9,996-element cell x 25 copies (320,000 of them refined): 1,490 ms with
// every pair by Gauss nodes in two-float arithmetic, 612 ms so (540 with the units dealt as below), with an
// error 10 to 25 times smaller
// (E: 2.0e-10 B before, 1.7e-11 B now, the largest of 665 refined points).  The FP32 pipe is busy for
// about two thirds of it; 5 blocks per SM (96 registers) beat 4 by 3 %, 6 are the same.
//
// Level 2 in the same run: 98 ms with every pair by Gauss nodes, 57 ms by moments (51); largest errors
// unchanged (phi 1.1e-15 B, E 1.1e-14 B).
//
// An element's sums over its images of one point (before sigma): Phi', and E' in the global frame.
struct ElemSum {
    double phi, x, y, z;
};
// The far pairs of a point (ph + pl) and element j of a staged tile at level L, of phi and E (M = kBoth),
// phi only or E only.
template <int L, int M>
__device__ __forceinline__ ElemSum acc_element(const AccView& A, int nimg, int np2, int64_t j, const FillEl& F,
                                               const float4* mom, const float4& hdr, const float* tau,
                                               const float (&ph)[3], const float (&pl)[3]) {
    // squared distance from which the moments are taken; never inside the near radius, which
    // the two classifications of a pair (here and in the near kernel) round differently
    constexpr double kRatio = L == 1 ? kMomRatio : kMomRatio2;
    const float mom2 = fmaxf(F.hdr.x * (float)(kRatio * kRatio / (kFillRatioA * kFillRatioA)), hdr.w * 1.0001f);
    float dh[3], dl[3];
    df_sub(ph[0], pl[0], F.ch.x, F.cl.x, dh[0], dl[0]);
    df_sub(ph[1], pl[1], F.ch.y, F.cl.y, dh[1], dl[1]);
    df_sub(ph[2], pl[2], F.ch.z, F.cl.z, dh[2], dl[2]);
    float x0h, x0l, y0h, y0l, z0h, z0l;
    df_dot3(dh, dl, F.exh, F.exl, x0h, x0l);
    df_dot3(dh, dl, F.eyh, F.eyl, y0h, y0l);
    df_dot3(dh, dl, F.ezh, F.ezl, z0h, z0l);
    MomSum2 S{};     // level 1
    PointSum2 S2{};  // level 2
    NearerSum nr{};
    bool any_nearer = false;
    uint32_t nearer = 0;  // images of the group of 32 at hand whose pair is not taken by moments
    for (int k = 0; k < np2; k += 2) {
        auto plane = [&](int q) { return *reinterpret_cast<const float2*>(tau + q * np2 + k); };
        // X = X0 - tau, two floats
        auto diff = [&](float ah, float al, int q, float2& h, float2& l) {
            float2 t;
            two_sum2(bc2(ah), plane(q), h, t);
            l = __fadd2_rn(t, __fadd2_rn(bc2(al), plane(q + 3)));
        };
        FillPair2 P;
        float2 &xh = P.xh, &xl = P.xl, &zh = P.zh, &zl = P.zl, yh, yl;
        diff(x0h, x0l, 0, xh, xl);
        diff(y0h, y0l, 1, yh, yl);
        diff(z0h, z0l, 2, zh, zl);
        float2 px = __fmul2_rn(xh, xh), py = __fmul2_rn(yh, yh), pz = __fmul2_rn(zh, zh);
        float2 ex = __ffma2_rn(xh, xh, make_float2(-px.x, -px.y)), ey = __ffma2_rn(yh, yh, make_float2(-py.x, -py.y)),
               ez = __ffma2_rn(zh, zh, make_float2(-pz.x, -pz.y));
        ex = __ffma2_rn(__fadd2_rn(xh, xh), xl, ex);
        ey = __ffma2_rn(__fadd2_rn(yh, yh), yl, ey);
        ez = __ffma2_rn(__fadd2_rn(zh, zh), zl, ez);
        float2 s, t1, t2, d2h;
        two_sum2(px, py, s, t1);
        two_sum2(s, pz, d2h, t2);
        const float2 d2l = __fadd2_rn(__fadd2_rn(ex, ey), __fadd2_rn(ez, __fadd2_rn(t1, t2)));
        const bool two = k + 1 < nimg;
        const bool far0 = d2h.x >= mom2, far1 = two && d2h.y >= mom2;
        if constexpr (L == 1) {
            mom_pair2<M != kEOnly, M != kPhiOnly>(mom, F.ch.w, xh, xl, yh, yl, zh, zl, d2h, d2l,
                                                  far0, far1, S);
        } else {
            P.px = px, P.ex = ex, P.pz = pz, P.ez = ez, P.d2h = d2h, P.d2l = d2l;
            fill_mom_point2(mom, P, yh, yl, far0, far1, S2);
        }
        nearer |= ((far0 ? 0u : 1u) | (far1 || !two ? 0u : 2u)) << (k & 31);
        if ((k & 31) == 30 || k + 2 >= np2) {
            for (uint32_t m = nearer; m; m &= m - 1) {
                const int kk = (k & ~31) + __ffs(m) - 1;
                acc_pair_nodes<M>(A, hdr, (int)F.hdr.w, j, nimg, kk, ph, pl, x0h, x0l, y0h, y0l, z0h, z0l, tau,
                                  np2, nr);
            }
            any_nearer = any_nearer || nearer;
            nearer = 0;
        }
    }
    // A x (sum over the images) + the other terms as two floats, then FP64, rotated to the global
    // frame.  A conversion takes the FP64 pipe like an addition does, so each quantity crosses over
    // once, as two values.
    ElemSum v{0.0, 0.0, 0.0, 0.0};
    double lx = 0.0, ly = 0.0, lz = 0.0;
    const float4 tail = mom[(L == 1 ? kMomF4 : kFillMomF4) - 1];
    if constexpr (L == 2) {
        auto area = [&](const float2& h, const float2& l, float nh, float nl) {  // A x + nearer
            float sh, t, p, e;
            two_sum(h.x, h.y, sh, t);
            const float sl = __fadd_rn(t, __fadd_rn(l.x, l.y));
            two_prod(sh, tail.x, p, e);
            e = __fmaf_rn(sh, tail.y, __fmaf_rn(sl, tail.x, e));
            double x = (double)p + (double)e;
            if (any_nearer) x += (double)nh + (double)nl;
            return x;
        };
        v.phi = area(S2.ph, S2.pl, nr.ph, nr.pl);
        lx = area(S2.xh, S2.xl, nr.xh, nr.xl);
        ly = area(S2.yh, S2.yl, nr.yh, nr.yl);
        lz = area(S2.zh, S2.zl, nr.zh, nr.zl);
    } else {
        // sign: -1 where the high parts are kept negated; unit: what c is kept over
        auto total = [&](float sign, float unit, const float2& h, const float2& l, const float2& c) {
            float sh, t, p, e;
            two_sum(h.x, h.y, sh, t);
            sh *= sign;
            const float sl = __fmaf_rn(sign, t, __fadd_rn(l.x, l.y));
            two_prod(sh, tail.z, p, e);
            e = __fmaf_rn(sh, tail.w, __fmaf_rn(sl, tail.z, e));
            return (double)p + (double)__fmaf_rn(__fadd_rn(c.x, c.y), unit, e);
        };
        const float rho = F.ch.w;
        if constexpr (M != kEOnly) {
            v.phi = total(1.f, rho * rho, S.ph, S.pl, S.fc);
            if (any_nearer) v.phi += (double)nr.ph + (double)nr.pl;
        }
        if constexpr (M != kPhiOnly) {
            lx = total(-1.f, rho, S.xh, S.xl, S.ex);
            ly = total(-1.f, rho, S.yh, S.yl, S.ey);
            lz = total(-1.f, rho, S.zh, S.zl, S.ez);
            if (any_nearer) {
                lx += (double)nr.xh + (double)nr.xl;
                ly += (double)nr.yh + (double)nr.yl;
                lz += (double)nr.zh + (double)nr.zl;
            }
        }
    }
    if constexpr (M != kPhiOnly) {
        const Elem& e = A.el[j];
        v.x = fma(lx, e.ex[0], fma(ly, e.ey[0], lz * e.ez[0]));
        v.y = fma(lx, e.ex[1], fma(ly, e.ey[1], lz * e.ez[1]));
        v.z = fma(lx, e.ex[2], fma(ly, e.ey[2], lz * e.ez[2]));
    }
    return v;
}

// Raw sums (before ke) over the elements [e0, e1) (at most a leaf) at level L, with the error
// scales; all threads of the block take part (tiles).
//   LANES = false: thread per point (ph + pl); returns its sums.
//   LANES = true: a thread per (point, element): warp w takes the points list[i0 + w kLP / 4 ...] of the
//   unit's kLP, te elements of 32 / te points at a time, and the ordered chains over the
//   elements follow from shared memory; the sums go to out[6 per point] in shared memory.
// Both give a point the same bits.
template <int L, int M, bool LANES>
__device__ __forceinline__ Sum6 acc_range(const AccView& A, int nimg, int te, float4* sm, float (&ph)[3], float (&pl)[3],
                                          int64_t e0, int64_t e1, const double* __restrict__ pts,
                                          const int32_t* __restrict__ list, int64_t i0, int64_t count) {
    constexpr int kMF4 = acc_mom_f4(L);
    const int np2 = acc_pad(nimg), ts = acc_tau_stride(nimg);
    FillEl* s_fe = reinterpret_cast<FillEl*>(sm);
    float4* s_mom = sm + 9 * te;
    float4* s_hdr = s_mom + kMF4 * te;
    float* s_tau = reinterpret_cast<float*>(s_hdr + te);
    LaneScratch* scr = reinterpret_cast<LaneScratch*>(sm + acc_tile_f4(L, te, nimg));
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    constexpr int kWP = kLP / (kAT / 32);  // points of a warp
    if constexpr (LANES) {
        for (int i = lane; i < 6 * kWP; i += 32) scr->out[w * kWP][i] = 0.0;
        __syncwarp();
    }
    const float4* gmom = L == 1 ? A.mom : A.mom2;
    constexpr int kGM = L == 1 ? kMomF4 : kFillMomF4;
    Sum6 acc{0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int64_t base = e0; base < e1; base += te) {
        const int cnt = (int)min((int64_t)te, e1 - base);
        __syncthreads();
        {
            const float4* src = reinterpret_cast<const float4*>(A.fe + base);
            float4* dst = reinterpret_cast<float4*>(s_fe);
            for (int i = threadIdx.x; i < 9 * cnt; i += blockDim.x) dst[i] = src[i];
        }
        for (int i = threadIdx.x; i < kGM * cnt; i += blockDim.x) s_mom[i / kGM * kMF4 + i % kGM] = gmom[base * kGM + i];
        for (int i = threadIdx.x; i < cnt; i += blockDim.x) {  // (-, tier a, tier b, FP64) squared radii
            const float4 f = A.fe[base + i].hdr;
            s_hdr[i] = L == 1 ? A.far[base + i].hdr : make_float4(0.f, f.x, f.y, f.z);
        }
        for (int i = threadIdx.x; i < cnt * np2; i += blockDim.x) {
            const int jj = i / np2, k = min(i - jj * np2, nimg - 1);
            const float4 h = A.tau[2 * ((base + jj) * nimg + k)], l = A.tau[2 * ((base + jj) * nimg + k) + 1];
            float* d = s_tau + jj * ts + (i - jj * np2);
            d[0] = -h.x, d[np2] = -h.y, d[2 * np2] = -h.z;
            d[3 * np2] = -l.x, d[4 * np2] = -l.y, d[5 * np2] = -l.z;
        }
        __syncthreads();
        const int per = 32 / te;  // points side by side (lanes)
        const int steps = LANES ? (kWP + per - 1) / per : cnt;
        for (int t = 0; t < steps; ++t) {
            const int jj = LANES ? lane % te : t;
            const int q = t * per + lane / te;  // LANES: the point of the warp's kWP
            bool valid = true;
            if constexpr (LANES) {
                const int64_t i = i0 + w * kWP + q;
                valid = jj < cnt && q < kWP && i < count;
                if (valid) load_point_2f(pts, list[i], true, ph[0], ph[1], ph[2], pl[0], pl[1], pl[2]);
            }
            double s = 0.0;
            ElemSum v{0.0, 0.0, 0.0, 0.0};
            if (valid) {
                s = A.sigma[base + jj];
                v = acc_element<L, M>(A, nimg, np2, base + jj, s_fe[jj], s_mom + kMF4 * jj, s_hdr[jj],
                                      s_tau + jj * ts, ph, pl);
            }
            if constexpr (!LANES) {
                if constexpr (M != kEOnly) {
                    acc.phi = fma(s, v.phi, acc.phi);
                    acc.bphi = fma(fabs(s), fabs(v.phi), acc.bphi);
                }
                if constexpr (M != kPhiOnly) {
                    acc.x = fma(s, v.x, acc.x);
                    acc.y = fma(s, v.y, acc.y);
                    acc.z = fma(s, v.z, acc.z);
                    acc.bE = fma(fabs(s), fabs(v.x) + fabs(v.y) + fabs(v.z), acc.bE);
                }
                continue;
            }
            LaneScratch::Val& o = scr->val[w][lane];
            o.d[0] = s, o.d[1] = v.phi, o.d[2] = v.x, o.d[3] = v.y, o.d[4] = v.z;
            o.a[0] = fabs(v.phi), o.a[1] = fabs(v.x) + fabs(v.y) + fabs(v.z);
            __syncwarp();
            // chain `which` (0 to 5) of a point by one lane, in the order of the elements
            const int m = min(per, kWP - t * per);
            for (int c = lane; c < 6 * m; c += 32) {
                const int qq = c / 6, which = c - 6 * qq;
                const LaneScratch::Val* r = scr->val[w] + qq * te;
                double& dst = scr->out[w * kWP + t * per + qq][which];
                double x = dst;
                const bool scale = which >= 4;
                for (int e = 0; e < cnt; ++e)
                    x = fma(scale ? fabs(r[e].d[0]) : r[e].d[0], scale ? r[e].a[which - 4] : r[e].d[1 + which], x);
                dst = x;
            }
            __syncwarp();
        }
    }
    return acc;
}

// ke * sums of point p at level L into phi / E, the level's estimate into err, and (level 1)
// ke * (B_phi, B_E, 0, 0) into bound for the next flag step; a quantity the pass does not
// re-evaluate (M) keeps its value and estimate, and its level-1 scale is 0, so that the
// next flag step does not take it up.
template <int L, int M>
__device__ __forceinline__ void store_acc(int64_t p, const Sum6& tot, double* __restrict__ phi,
                                          double* __restrict__ E, double* __restrict__ err,
                                          float4* __restrict__ bound) {
    const double ke = 1.0 / (4.0 * kPi * kEps0);
    const double gamma = (L == 1) ? kGammaL1 : kGammaL2;
    if (M != kEOnly && phi) phi[p] = ke * tot.phi;
    if (M != kPhiOnly && E) {
        E[3 * p] = ke * tot.x;
        E[3 * p + 1] = ke * tot.y;
        E[3 * p + 2] = ke * tot.z;
    }
    if (err) {
        if (M != kEOnly) err[2 * p] = gamma * ke * tot.bphi;
        if (M != kPhiOnly) err[2 * p + 1] = gamma * ke * tot.bE;
    }
    if (L == 1)
        bound[p] = make_float4(M != kEOnly ? (float)(ke * tot.bphi) : 0.f, M != kPhiOnly ? (float)(ke * tot.bE) : 0.f,
                               0.f, 0.f);
}

// The far sums of one point over whole pieces of the summation tree.
template <int L, int M>
__device__ __forceinline__ Sum6 acc_sum(const AccView& A, int nimg, int te, float4* sm, float (&ph)[3],
                                        float (&pl)[3], int64_t e0, int64_t e1) {
    Sum6 tot{0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int64_t c0 = e0; c0 < e1; c0 += kChunkEl) {
        const int64_t c1 = min(c0 + (int64_t)kChunkEl, e1);
        Sum6 ch{0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        for (int64_t l = c0; l < c1; l += kLeafEl)
            add_sum(ch, acc_range<L, M, false>(A, nimg, te, sm, ph, pl, l, min(l + (int64_t)kLeafEl, c1), nullptr,
                                               nullptr, 0, 0));
        add_sum(tot, ch);
    }
    return tot;
}

// Far part of every listed point at level L, thread per point, kAT points (a group) per
// block pass.  The ceil(*n_list / kAT) groups are dealt by split_plan: whole groups, then the
// pieces of the left-over groups, whose Sum6 go to part[(i - Gm kAT) np + piece] of list entry
// i for k_acc_reduce.  The resident blocks take the units in turn as they finish (*next): dealt round
// robin, 15 of 20 warps per SM were there on average, since units near the points take longer (1e6
// points: level 1 612 ms, level 2 57; in turn 540 and 51).  A point gets the same bits whichever way it is taken.  M: which
// quantities the pass re-evaluates (kBoth, kPhiOnly, kEOnly).
template <int L, int M>
__global__ void __launch_bounds__(kAT, kATBlocks)
    k_eval_acc_far(const AccView A, int nimg, int te, const double* __restrict__ pts,
                   const int32_t* __restrict__ list, const int32_t* __restrict__ n_list, int32_t* next, int64_t gb,
                   int64_t cap, Sum6* __restrict__ part, double* __restrict__ phi, double* __restrict__ E,
                   double* __restrict__ err, float4* __restrict__ bound) {
    extern __shared__ float4 sm[];
    const int64_t count = *n_list;
    const SplitPlan plan = split_plan((count + kAT - 1) / kAT, gb, A.n_el, cap);
    if (lane_path(plan, count, gb)) return;
    const int64_t units = plan.Gm + plan.R * plan.np;
    __shared__ int s_unit;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_unit = atomicAdd(next, 1);
        __syncthreads();
        const int64_t u = s_unit;
        if (u >= units) break;
        const SplitUnit t = split_unit(plan, u, A.n_el);
        const int64_t i = t.group * kAT + threadIdx.x;
        const bool active = i < count;
        const int64_t p = active ? (int64_t)list[i] : 0;
        float ph[3], pl[3];
        load_point_2f(pts, p, active, ph[0], ph[1], ph[2], pl[0], pl[1], pl[2]);
        const Sum6 tot = acc_sum<L, M>(A, nimg, te, sm, ph, pl, t.e0, t.e1);
        if (!active) continue;
        if (t.whole)
            store_acc<L, M>(p, tot, phi, E, err, bound);
        else
            part[(t.r * kAT + threadIdx.x) * plan.np + t.piece] = tot;
    }
}

// The same for short lists (lane_path): a unit is kLP points of one leaf, a thread takes (point, element)
// pairs, and the leaf's sums go to the same partial sums.
template <int L, int M>
__global__ void __launch_bounds__(kAT, 4)
    k_eval_acc_lanes(const AccView A, int nimg, int te, const double* __restrict__ pts,
                     const int32_t* __restrict__ list, const int32_t* __restrict__ n_list, int64_t gb,
                     int64_t cap, Sum6* __restrict__ part) {
    extern __shared__ float4 sm[];
    const int64_t count = *n_list;
    const SplitPlan plan = split_plan((count + kAT - 1) / kAT, gb, A.n_el, cap);
    if (!lane_path(plan, count, gb)) return;
    const int64_t lg = (count + kLP - 1) / kLP;
    const LaneScratch* scr = reinterpret_cast<LaneScratch*>(sm + acc_tile_f4(L, te, nimg));
    constexpr int kWP = kLP / (kAT / 32);
    const int w = threadIdx.x >> 5;
    for (int64_t u = blockIdx.x; u < lg * plan.np; u += gridDim.x) {
        const int64_t piece = u / lg, i0 = (u - piece * lg) * kLP;  // consecutive units: the same leaf
        const int64_t e0 = piece * kLeafEl;
        float ph[3], pl[3];
        acc_range<L, M, true>(A, nimg, te, sm, ph, pl, e0, min(e0 + (int64_t)kLeafEl, A.n_el), pts, list, i0, count);
        for (int c = threadIdx.x & 31; c < 6 * kWP; c += 32) {
            const int64_t q = i0 + w * kWP + c / 6;
            if (q < count) reinterpret_cast<double*>(part + q * plan.np + piece)[c % 6] = scr->out[w * kWP + c / 6][c % 6];
        }
        __syncwarp();
    }
}

// The left-over groups of k_eval_acc_far: their pieces added along the summation tree, a warp
// per point.
template <int L, int M>
__global__ void __launch_bounds__(256)
    k_acc_reduce(int64_t n_el, const int32_t* __restrict__ list, const int32_t* __restrict__ n_list, int64_t gb,
                 int64_t cap, const Sum6* __restrict__ part, double* __restrict__ phi, double* __restrict__ E,
                 double* __restrict__ err, float4* __restrict__ bound) {
    const int64_t count = *n_list;
    const SplitPlan plan = split_plan((count + kAT - 1) / kAT, gb, n_el, cap);
    const int64_t first = plan.Gm * kAT, warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; first + w < count; w += warps) {
        const Sum6 tot = split_reduce(part + w * plan.np, plan.np, plan.leaf);
        if ((threadIdx.x & 31) == 0) store_acc<L, M>(list[first + w], tot, phi, E, err, bound);
    }
}

// FP64 near pairs of every listed point, a warp per point (near_point_warp): level 1 with
// the FP32 pass's near radii, level 2 with the fill's.
template <int L>
__global__ void __launch_bounds__(kAT)
    k_eval_acc_near(const AccView A, const ImageTable img, const double* __restrict__ pts,
                    const int32_t* __restrict__ list, const int32_t* __restrict__ n_list, double* __restrict__ phi,
                    double* __restrict__ E) {
    __shared__ int32_t s_queue[kAT / 32][kNearQueue];
    const int64_t count = *n_list, warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < count; w += warps) {
        if constexpr (L == 1)
            near_point_warp(A.el, A.sigma, A.cjk, A.view.grid, A.view.cell_start, A.view.cell_items, img,
                            NearFar{A.far}, pts, list[w], phi, E, s_queue[threadIdx.x >> 5]);
        else
            near_point_warp(A.el, A.sigma, A.cjk, A.grid, A.cell_start, A.cell_items, img, NearFill{A.fe}, pts,
                            list[w], phi, E, s_queue[threadIdx.x >> 5]);
    }
}

// Flags and lists (in their input order within each block) the points whose estimate
// gr |x| + gb B + gs S (x = phi or E, bound = (B_phi, B_E, S_phi, S_E)) exceeds tol |x| (when
// refine != 0): with sel < 0 every such point; with sel = kBoth, kPhiOnly or kEOnly the
// points where both quantities, phi only or E only exceed it.  Input: order[i] (or i when
// order is null) for i < n, or i < *n_dev when n_dev is given.  err (may be null) receives
// every input point's estimate.
__global__ void __launch_bounds__(256)
    k_flag(const double* __restrict__ phi, const double* __restrict__ E, const float4* __restrict__ bound,
           const int32_t* __restrict__ order, int64_t n, const int32_t* __restrict__ n_dev, double gr, double gb,
           double gs, double tol, int refine, int sel, double* __restrict__ err, int32_t* __restrict__ list,
           int32_t* __restrict__ n_list) {
    __shared__ int32_t s_warp[8];
    __shared__ int32_t s_base;
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int64_t count = n_dev ? (int64_t)*n_dev : n;
    bool f = false;
    int32_t p = 0;
    if (i < count) {
        p = order ? order[i] : (int32_t)i;
        const float4 b = bound[p];
        const double ap = phi ? fabs(phi[p]) : 0.0;
        double aE = 0.0;
        if (E) {
            const double ex = E[3 * p], ey = E[3 * p + 1], ez = E[3 * p + 2];
            aE = sqrt(ex * ex + ey * ey + ez * ez);
        }
        const double ep = gr * ap + gb * (double)b.x + gs * (double)b.z;
        const double eE = gr * aE + gb * (double)b.y + gs * (double)b.w;
        const bool fp = phi && ep > tol * ap, fe = E && eE > tol * aE;
        const int mode = (fp && fe) ? kBoth : fp ? kPhiOnly : kEOnly;
        f = refine && (fp || fe) && (sel < 0 || sel == mode);
        if (err) {
            err[2 * p] = ep;
            err[2 * p + 1] = eE;
        }
    }
    const unsigned ballot = __ballot_sync(0xffffffffu, f);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) s_warp[w] = __popc(ballot);
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t run = 0;
        for (int k = 0; k < 8; ++k) {
            const int32_t c = s_warp[k];
            s_warp[k] = run;
            run += c;
        }
        s_base = run ? atomicAdd(n_list, run) : 0;
    }
    __syncthreads();
    if (f) list[s_base + s_warp[w] + __popc(ballot & ((1u << lane) - 1u))] = p;
}

template <int L, int M>
cudaError_t launch_level(const AccView& A, const ImageTable& img, const double* pts, int64_t npts, double* phi,
                         double* E, double* err, float4* bound, const int32_t* list, const int32_t* n_list,
                         int32_t* next, int sms, Sum6* part, int64_t cap, cudaStream_t s) {
    // element tile: a power of two (divides the leaf), within ~40 KB
    constexpr int kSmem = 40 * 1024;
    int te = kLeafEl;
    while (te > 1 && acc_tile_f4(L, te, img.n) * (int)sizeof(float4) > kSmem) te /= 2;
    const size_t smem = (size_t)acc_tile_f4(L, te, img.n) * sizeof(float4), lane_smem = smem + sizeof(LaneScratch);
    const int64_t gb = kATBlocks * (int64_t)sms, want = (npts + kAT - 1) / kAT;
    cudaError_t e;
    // the list's length is known on the device: both kernels are launched unless even the whole input is short
    if (!lane_path(split_plan(want, gb, A.n_el, cap), npts, gb)) {
        // one value whatever the tile: another thread's call may be between this and its launch
        e = cudaFuncSetAttribute(k_eval_acc_far<L, M>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
        if (e != cudaSuccess) return e;
        const int64_t most = want * split_count(A.n_el, kLeafEl);  // units of the longest list
        k_eval_acc_far<L, M><<<(unsigned)std::min(gb, most), kAT, smem, s>>>(A, img.n, te, pts, list, n_list, next, gb,
                                                                            cap, part, phi, E, err, bound);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    e = cudaFuncSetAttribute(k_eval_acc_lanes<L, M>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kSmem + (int)sizeof(LaneScratch));
    if (e != cudaSuccess) return e;
    k_eval_acc_lanes<L, M><<<(unsigned)std::min<int64_t>(4 * (int64_t)sms, split_count(npts, kLP) * split_count(A.n_el, kLeafEl)),
                             kAT, lane_smem, s>>>(A, img.n, te, pts, list, n_list, gb, cap, part);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int64_t left = std::min(want, 2 * gb) * kAT;  // points of the left-over groups, at most
    k_acc_reduce<L, M><<<(unsigned)std::min<int64_t>((left + 7) / 8, 8 * (int64_t)sms), 256, 0, s>>>(
        A.n_el, list, n_list, gb, cap, part, phi, E, err, bound);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // the FP64 near pairs, added to the quantities this pass re-evaluated only
    double* nphi = (M == kEOnly) ? nullptr : phi;
    double* nE = (M == kPhiOnly) ? nullptr : E;
    const unsigned gn = (unsigned)std::min<int64_t>((npts + kAT / 32 - 1) / (kAT / 32), 16 * (int64_t)sms);
    k_eval_acc_near<L><<<gn, kAT, 0, s>>>(A, img, pts, list, n_list, nphi, nE);
    return cudaGetLastError();
}

// ElemMom records (twofloat.cuh) from the elements' 36-node rules, which integrate degree 4 exactly.
__global__ void k_elem_moments(const FillEl* __restrict__ fe, const float4* __restrict__ nodes, int64_t n,
                               float4* __restrict__ mom) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const float4* nd = nodes + j * kFillNodeRec + kFillOffC;
    const double half = -0.5 / (double)fe[j].ch.w;  // u = (node - centroid) / rho = -s / rho, stored as 2 s
    double A = 0.0, M2[3] = {}, M3[4] = {}, M4[5] = {};
    for (int q = 0; q < kFillPairsC; ++q) {
        const float4 h0 = nd[4 * q], h1 = nd[4 * q + 1], l0 = nd[4 * q + 2], l1 = nd[4 * q + 3];
        for (int lane = 0; lane < 2; ++lane) {
            const double x = half * (lane ? (double)h0.y + (double)l0.y : (double)h0.x + (double)l0.x);
            const double z = half * (lane ? (double)h0.w + (double)l0.w : (double)h0.z + (double)l0.z);
            const double w = lane ? (double)h1.w + (double)l1.w : (double)h1.z + (double)l1.z;
            A += w;
            M2[0] += w * x * x, M2[1] += w * x * z, M2[2] += w * z * z;
            M3[0] += w * x * x * x, M3[1] += w * x * x * z, M3[2] += w * x * z * z, M3[3] += w * z * z * z;
            M4[0] += w * x * x * x * x, M4[1] += w * x * x * x * z, M4[2] += w * x * x * z * z;
            M4[3] += w * x * z * z * z, M4[4] += w * z * z * z * z;
        }
    }
    const double t2 = M2[0] + M2[2], q0 = 0.375 * (M4[0] + 2 * M4[2] + M4[4]);
    const double c[22] = {3 * M2[0], 3 * M2[1], 3 * M2[2], -0.5 * t2,
                          7.5 * M3[0], 7.5 * M3[1], 7.5 * M3[2], 7.5 * M3[3],
                          -1.5 * (M3[0] + M3[2]), -1.5 * (M3[1] + M3[3]),
                          17.5 * M4[0], 17.5 * M4[1], 17.5 * M4[3], 17.5 * M4[4], 52.5 * M4[1], 52.5 * M4[2],
                          52.5 * M4[3], -7.5 * (M4[0] + M4[2]), -7.5 * (M4[1] + M4[3]), -7.5 * (M4[2] + M4[4]),
                          q0, 5 * q0};
    float4* out = mom + j * kMomF4;
    for (int q = 0; q < kMomF4 - 1; ++q) {
        const float a = (float)c[2 * q], b = (float)c[2 * q + 1];
        out[q] = make_float4(a, a, b, b);
    }
    const float t3 = (float)(-1.5 * t2), ah = (float)A;
    out[kMomF4 - 1] = make_float4(t3, t3, ah, (float)(A - (double)ah));
}

}  // namespace

size_t elem_moments_bytes(int64_t n) { return sizeof(float4) * kMomF4 * (size_t)n; }
cudaError_t launch_elem_moments(const FillEl* fe, const float4* nodes, int64_t n, float4* mom, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_elem_moments<<<(unsigned)((n + 63) / 64), 64, 0, s>>>(fe, nodes, n, mom);
    return cudaGetLastError();
}

ErrModel default_err_model() { return ErrModel{kErrGammaR, kErrGammaB, kErrGammaS}; }

size_t refine_part_bytes(int64_t npts, int sms, int64_t n_el) {
    static_assert(kAT == kEvalThreads, "points of a group");
    return split_part_bytes<Sum6>(npts, kATBlocks * (int64_t)sms, n_el);
}

cudaError_t launch_eval_refine(const AccView& A, const ImageTable& img, const double* pts, int64_t npts,
                               double* phi, double* E, double* err, double tol, const ErrModel& em,
                               const MixedScratch& ms, int sms, cudaStream_t s, cudaEvent_t* ev, void* part_buf,
                               size_t part_bytes) {
    Sum6* part = static_cast<Sum6*>(part_buf);
    const int64_t cap = (int64_t)(part_bytes / sizeof(Sum6));
    if (npts == 0) return cudaSuccess;
    if (npts > (int64_t)INT32_MAX) return cudaErrorInvalidValue;
    const bool refine = tol > 0.0 && (phi || E);
    // counts: [0] level 1, both quantities; [1] level 2; [2] level 1, phi only; [3] level 1, E only;
    // [4] to [7] the next unit of the passes
    cudaError_t e = cudaMemsetAsync(ms.n_list, 0, kRefineCounts * sizeof(int32_t), s);
    if (e != cudaSuccess) return e;
    const unsigned fb = (unsigned)((npts + 255) / 256);
    k_flag<<<fb, 256, 0, s>>>(phi, E, ms.bound, ms.order, npts, nullptr, em.gamma_r, em.gamma_b, em.gamma_s, tol,
                              refine ? 1 : 0, kBoth, err, ms.list, ms.n_list);
    e = cudaGetLastError();
    // level 1 on the flagged points, in three passes by what they need (warps then hold
    // points of one kind); it leaves their level-1 scales in ms.bound
    if (e == cudaSuccess && refine) {
        k_flag<<<fb, 256, 0, s>>>(phi, E, ms.bound, ms.order, npts, nullptr, em.gamma_r, em.gamma_b, em.gamma_s,
                                  tol, 1, kPhiOnly, nullptr, ms.list_p, ms.n_list + 2);
        k_flag<<<fb, 256, 0, s>>>(phi, E, ms.bound, ms.order, npts, nullptr, em.gamma_r, em.gamma_b, em.gamma_s,
                                  tol, 1, kEOnly, nullptr, ms.list_e, ms.n_list + 3);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && refine)
        e = launch_level<1, kBoth>(A, img, pts, npts, phi, E, err, ms.bound, ms.list, ms.n_list, ms.n_list + 4, sms, part,
                                    cap, s);
    if (e == cudaSuccess && refine)
        e = launch_level<1, kPhiOnly>(A, img, pts, npts, phi, E, err, ms.bound, ms.list_p, ms.n_list + 2, ms.n_list + 5, sms,
                                      part, cap, s);
    if (e == cudaSuccess && refine)
        e = launch_level<1, kEOnly>(A, img, pts, npts, phi, E, err, ms.bound, ms.list_e, ms.n_list + 3, ms.n_list + 6, sms,
                                    part, cap, s);
    if (e == cudaSuccess && ev) e = cudaEventRecord(ev[0], s);
    if (e == cudaSuccess && refine) {
        // level 2 on the points whose level-1 estimate still exceeds the tolerance (a quantity
        // that level 1 left alone has a level-1 scale of 0 and is not taken up again)
        const int32_t* l1[3] = {ms.list, ms.list_p, ms.list_e};
        const int32_t* c1[3] = {ms.n_list, ms.n_list + 2, ms.n_list + 3};
        for (int k = 0; k < 3; ++k)
            k_flag<<<fb, 256, 0, s>>>(phi, E, ms.bound, l1[k], npts, c1[k], 0.0, kGammaL1, 0.0, tol, 1, -1, nullptr,
                                      ms.list2, ms.n_list + 1);
        e = cudaGetLastError();
        if (e == cudaSuccess)
            e = launch_level<2, kBoth>(A, img, pts, npts, phi, E, err, nullptr, ms.list2, ms.n_list + 1, ms.n_list + 7, sms,
                                    part, cap, s);
    }
    if (e == cudaSuccess && ev) e = cudaEventRecord(ev[1], s);
    return e;
}

}  // namespace nb
