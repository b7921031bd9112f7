// influence.cuh -- closed-form potential and field of a uniformly charged flat polygon
// (rectangle or triangle), FP64, device code.
//
// Sec. 2.1 defines Phi'(P) = int_S dA / |P - r'| and E'(P) = int_S (P - r') dA / |P - r'|^3
// over a flat rectangle or triangle.  Both shapes are evaluated here with one boundary
// decomposition of the surface integral.  The target P has local coordinates
// (X, Y, Z); the element lies in the plane y = 0 with counter-clockwise vertices
// q_i = (qx_i, qz_i).  Per edge i (q_i -> q_i+1, unit tangent t, outward normal m):
//   d_i   signed distance from the projection (X, Z) to the edge line (inside > 0),
//   L_i = int_edge dl / R = ln((R+ + l+) / (R- + l-)),   l-/+ tangential end coordinates,
// and with Omega the solid angle subtended by the element (signed like Y):
//   Phi'  = sum_i d_i L_i - Y Omega,
//   E'_xz = sum_i m_i L_i            (in-plane part: surface gradient -> boundary term),
//   E'_y  = Omega                    (normal part).
// Omega is summed over the fan triangles (0,1,2) and (0,2,3) with the Van Oosterom -
// Strackee form tan(Omega/2) = N / D, N = 2A Y, D = R0 R1 R2 + (r0.r1) R2 + (r0.r2) R1
// + (r1.r2) R0 -- the numerator is exact (doubled area times height), so the far field
// of the normal component suffers no cancellation.  The two half-angles of a four-sided
// element are added as the argument of the product (D1 + i N1)(D2 + i N2) (one atan2).  Within 1e-4 element radii of the
// plane the solid angle is instead summed over the triangles (projection, q_i, q_i+1),
// which stays well-conditioned where the projection meets the fan diagonal.  Exactly in
// the element's plane (Y == 0) the normal field is the principal value 0.
//
// ln(l + R) with l < 0 cancels; the three cases below pick a cancellation-free ratio:
//   l- >= 0 :  (l+ + R+) / (l- + R-)
//   l+ <= 0 :  (R- - l-) / (R+ - l+)
//   else    :  (l+ + R+)(R- - l-) / rho^2,   rho^2 = d^2 + Y^2.
//
// Far from the element (every edge seen from more than about 3.5 of its lengths: len_i / (R_i
// + R_i+1) < 1/8 for all i) the same closed form is evaluated through
//   L_i = 2 artanh(x_i),  x_i = len_i / (R_i + R_i+1),     Omega = 2 arctan(N / D),
// with polynomials in x_i^2 and (N / D)^2 in place of log and atan2, and with the roots and
// quotients from one third-order step on the hardware's estimates (nr_sqrt, nr_div): 114
// FP64 instructions for a triangle and 155 for a quadrilateral against the 278 a pair (mean)
// of the general form, on a pipe of two FP64 operations per SM and clock that nothing else
// competes for.  It is also the more accurate form there: L_i is small, and the logarithm of a
// ratio near 1 keeps only the ratio's absolute rounding error (relative error 2^-53 / x_i).
// Every operation of both forms is an explicitly rounded intrinsic, so that the compiler's
// choice of contractions cannot make two kernels differ.
#pragma once
#include "nb_internal.h"

namespace nb {

// 1 / sqrt(x) of a normal FP32 number: rsqrtf without its scaling of subnormal arguments (the same bits).
__device__ __forceinline__ float rsqrt_normal(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// sqrt(a) for a normal a > 0: one third-order Householder step, a (y (1 + e/2 + 3 e^2/8)) with
// e = 1 - a y^2, on the hardware's estimate y of 1 / sqrt(a) (about 20 bits, so the step
// leaves the rounding of the last operations).  NaN for a = 0.
__device__ __forceinline__ double nr_sqrt(double a) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
    const double t = __dmul_rn(a, y);
    const double e = __fma_rn(-t, y, 1.0);
    return __fma_rn(t, __dmul_rn(__fma_rn(e, 0.375, 0.5), e), t);
}
// a / b for normal operands and quotient: a y (1 + e + e^2) with e = 1 - b y on the estimate y
// of 1 / b.  NaN for b = 0.
__device__ __forceinline__ double nr_div(double a, double b) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
    const double e = __fma_rn(-b, y, 1.0);
    const double t = __dmul_rn(a, y);
    return __fma_rn(t, __fma_rn(e, e, e), t);
}

// 2 artanh(x) / x as a polynomial in u = x^2 <= 1/64: the Taylor series economised with
// Chebyshev polynomials on that interval (relative error 4.2e-18).
__device__ __forceinline__ double artanh2_poly(double u) {
    double p = 0x1.4a764ef7b2eacp-3;
    p = __fma_rn(p, u, 0x1.7407a240e474ap-3);
    p = __fma_rn(p, u, 0x1.c71d5bfe7ca28p-3);
    p = __fma_rn(p, u, 0x1.2492488022531p-2);
    p = __fma_rn(p, u, 0x1.9999999a07711p-2);
    p = __fma_rn(p, u, 0x1.5555555555479p-1);
    return __fma_rn(p, u, 2.0);
}
// The same for u <= 1/4 (relative error 1.3e-17): the middle distances, x_i < 1/2.
__device__ __forceinline__ double artanh2_poly_mid(double u) {
    double p = 0x1.ce48b9be17d03p-2;
    p = __fma_rn(p, u, -0x1.3c7161316f0d8p-2);
    p = __fma_rn(p, u, 0x1.2b53fe10b0c42p-2);
    p = __fma_rn(p, u, 0x1.cb5b382cd4689p-6);
    p = __fma_rn(p, u, 0x1.eb5f578307cf7p-4);
    p = __fma_rn(p, u, 0x1.d8c89c0a1f0c0p-4);
    p = __fma_rn(p, u, 0x1.118bc9b54010ep-3);
    p = __fma_rn(p, u, 0x1.3b0abe34e132bp-3);
    p = __fma_rn(p, u, 0x1.745d881bea145p-3);
    p = __fma_rn(p, u, 0x1.c71c6e30d9d28p-3);
    p = __fma_rn(p, u, 0x1.2492492d4a1e8p-2);
    p = __fma_rn(p, u, 0x1.999999998388ep-2);
    p = __fma_rn(p, u, 0x1.5555555555605p-1);
    return __fma_rn(p, u, 2.0);
}
// 2 arctan(t) / t in u = t^2: Taylor series to u^5.  In the far form Omega <= len^2 / (3.4
// len)^2, so |t| = tan(Omega / 2) <= 0.044 and the first term left out is 3e-18.
__device__ __forceinline__ double arctan2_poly(double u) {
    double p = -2.0 / 11.0;
    p = __fma_rn(p, u, 2.0 / 9.0);
    p = __fma_rn(p, u, -2.0 / 7.0);
    p = __fma_rn(p, u, 2.0 / 5.0);
    p = __fma_rn(p, u, -2.0 / 3.0);
    return __fma_rn(p, u, 2.0);
}

// What the far form takes beside Elem, made once per element and block: unit tangents and
// lengths of the edges.
struct PolyEdges {
    double tx[4], tz[4], len[4];
};
__device__ __forceinline__ void poly_edge(const Elem& e, int i, PolyEdges& g) {
    const int j = (i + 1 == e.nv) ? 0 : i + 1;
    const double dx = e.qx[j] - e.qx[i], dz = e.qz[j] - e.qz[i];
    g.tx[i] = dx * e.inv_len[i];
    g.tz[i] = dz * e.inv_len[i];
    g.len[i] = __fma_rn(dx, g.tx[i], __dmul_rn(dz, g.tz[i]));
}

// The general form, at any place.
template <int NV>
__device__ __noinline__ void poly_general(const Elem& e, double X, double Y, double Z, double& phi, double& Ex,
                                          double& Ey, double& Ez) {
    double ax[NV], az[NV], R[NV];
    const double Y2 = __dmul_rn(Y, Y);
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        ax[i] = __dsub_rn(e.qx[i], X);
        az[i] = __dsub_rn(e.qz[i], Z);
        R[i] = sqrt(__fma_rn(ax[i], ax[i], __fma_rn(az[i], az[i], Y2)));
    }
    double sphi = 0.0, sx = 0.0, sz = 0.0;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const int j = (i + 1 == NV) ? 0 : i + 1;
        const double il = e.inv_len[i];
        const double tx = __dmul_rn(__dsub_rn(e.qx[j], e.qx[i]), il);
        const double tz = __dmul_rn(__dsub_rn(e.qz[j], e.qz[i]), il);
        const double d = __fma_rn(ax[i], tz, -__dmul_rn(az[i], tx));
        const double lm = __fma_rn(ax[i], tx, __dmul_rn(az[i], tz));
        const double lp = __fma_rn(ax[j], tx, __dmul_rn(az[j], tz));
        const double rho2 = __fma_rn(d, d, Y2);
        const bool pos = lm >= 0.0;
        const bool neg = lp <= 0.0;
        const double a = __dadd_rn(lp, R[j]);
        const double b = __dsub_rn(R[i], lm);
        const double num = pos ? a : (neg ? b : __dmul_rn(a, b));
        const double den = pos ? __dadd_rn(lm, R[i]) : (neg ? __dsub_rn(R[j], lp) : rho2);
        const double L = log(num / den);
        sphi = __dadd_rn(sphi, (d != 0.0) ? __dmul_rn(d, L) : 0.0);
        sx = __fma_rn(tz, L, sx);
        sz = __fma_rn(-tx, L, sz);
    }
    double om = 0.0;
    if (Y != 0.0) {
        if (fabs(Y) >= 1e-4 * e.rho) {
            // half-angles of the fan triangles as arguments of D + i N; their sum is the
            // argument of the product, which stays inside (-pi, pi) here (the element
            // subtends less than a hemisphere by a margin of order 1e-4), so one atan2
            // of the product replaces one per triangle
            double re = 1.0, im = 0.0;
#pragma unroll
            for (int f = 0; f < NV - 2; ++f) {
                const int i1 = f + 1, i2 = f + 2;
                const double d01 = __fma_rn(ax[0], ax[i1], __fma_rn(az[0], az[i1], Y2));
                const double d02 = __fma_rn(ax[0], ax[i2], __fma_rn(az[0], az[i2], Y2));
                const double d12 = __fma_rn(ax[i1], ax[i2], __fma_rn(az[i1], az[i2], Y2));
                const double D = __fma_rn(__dmul_rn(R[0], R[i1]), R[i2],
                                          __fma_rn(d01, R[i2], __fma_rn(d02, R[i1], __dmul_rn(d12, R[0]))));
                const double Nf = __dmul_rn(e.twoA[f], Y);
                if (f == 0) {
                    re = D;
                    im = Nf;
                } else {
                    const double r2 = __fma_rn(re, D, -__dmul_rn(im, Nf));
                    im = __fma_rn(re, Nf, __dmul_rn(im, D));
                    re = r2;
                }
            }
            om = 2.0 * atan2(im, re);
        } else {
            // Close to the plane the fan split is ill-conditioned where the projection
            // meets the shared diagonal; split at the projection instead: triangle
            // (p0, q_i, q_i+1) per edge, tan(Omega_i / 2) = sign(Y) c_i / (R_i R_j +
            // |Y| (R_i + R_j) + r_i . r_j) with c_i the doubled signed area.
            const double h = fabs(Y);
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                const int j = (i + 1 == NV) ? 0 : i + 1;
                const double cr = __fma_rn(ax[i], az[j], -__dmul_rn(az[i], ax[j]));
                const double dij = __fma_rn(ax[i], ax[j], __fma_rn(az[i], az[j], Y2));
                const double D = __fma_rn(R[i], R[j], __fma_rn(h, __dadd_rn(R[i], R[j]), dij));
                om = __dadd_rn(om, 2.0 * atan2(cr, D));
            }
            om = (Y > 0.0) ? om : -om;
        }
    }
    phi = __fma_rn(-Y, om, sphi);
    Ex = sx;
    Ey = om;
    Ez = sz;
}

// The far form where every x_i < 1/8 and, with a longer polynomial and atan2, where every
// x_i < 1/2; the general one else (nearer, or where an operand of the estimates is zero or not
// finite, which leaves a NaN x_i: a point on a vertex, or one without a place).  x_i < 1/2 on
// every edge keeps the projection outside the element wherever the height is small, so that
// D > 0 and the fan needs no care near the plane.  Without the middle distances the cube's solve
// and map (many pairs at 2 to 4 edge lengths) was 5 % slower than with the general form alone.
// kPhi, kField: which results are wanted (the others are left alone).
constexpr unsigned kEighthHi = 0x3fc00000u;  // high words of 1/8 and 1/2: positive doubles order as their words
constexpr unsigned kHalfHi = 0x3fe00000u;

template <int NV, bool kPhi, bool kField>
__device__ __forceinline__ void poly_f64(const Elem& e, const PolyEdges& g, double X, double Y, double Z, double& phi,
                                         double& Ex, double& Ey, double& Ez) {
    double ax[NV], az[NV], R[NV], x[NV];
    const double Y2 = __dmul_rn(Y, Y);
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        ax[i] = __dsub_rn(e.qx[i], X);
        az[i] = __dsub_rn(e.qz[i], Z);
        R[i] = nr_sqrt(__fma_rn(ax[i], ax[i], __fma_rn(az[i], az[i], Y2)));
    }
    unsigned worst = 0;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        x[i] = nr_div(g.len[i], __dadd_rn(R[i], R[i + 1 == NV ? 0 : i + 1]));
        worst = max(worst, (unsigned)__double2hiint(x[i]));  // a NaN of either sign is above every number
    }
    if (worst >= kHalfHi) {
        double f, gx, gy, gz;
        poly_general<NV>(e, X, Y, Z, f, gx, gy, gz);
        if constexpr (kPhi) phi = f;
        if constexpr (kField) {
            Ex = gx;
            Ey = gy;
            Ez = gz;
        }
        return;
    }
    const bool far = worst < kEighthHi;
#pragma unroll
    for (int i = 0; i < NV; ++i) {  // x_i becomes L_i
        const double u = __dmul_rn(x[i], x[i]);
        x[i] = __dmul_rn(x[i], far ? artanh2_poly(u) : artanh2_poly_mid(u));
    }
    double sphi = 0.0, sx = 0.0, sz = 0.0;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const double L = x[i];
        if constexpr (kPhi) {
            const double d = __fma_rn(ax[i], g.tz[i], -__dmul_rn(az[i], g.tx[i]));
            sphi = __fma_rn(d, L, sphi);
        }
        if constexpr (kField) {
            sx = __fma_rn(g.tz[i], L, sx);
            sz = __fma_rn(-g.tx[i], L, sz);
        }
    }
    double re = 1.0, im = 0.0;
#pragma unroll
    for (int f = 0; f < NV - 2; ++f) {
        const int i1 = f + 1, i2 = f + 2;
        const double d01 = __fma_rn(ax[0], ax[i1], __fma_rn(az[0], az[i1], Y2));
        const double d02 = __fma_rn(ax[0], ax[i2], __fma_rn(az[0], az[i2], Y2));
        const double d12 = __fma_rn(ax[i1], ax[i2], __fma_rn(az[i1], az[i2], Y2));
        const double D = __fma_rn(__dmul_rn(R[0], R[i1]), R[i2],
                                  __fma_rn(d01, R[i2], __fma_rn(d02, R[i1], __dmul_rn(d12, R[0]))));
        const double Nf = __dmul_rn(e.twoA[f], Y);
        if (f == 0) {
            re = D;
            im = Nf;
        } else {
            const double r2 = __fma_rn(re, D, -__dmul_rn(im, Nf));
            im = __fma_rn(re, Nf, __dmul_rn(im, D));
            re = r2;
        }
    }
    double om;
    if (far) {
        const double t = nr_div(im, re);
        om = __dmul_rn(t, arctan2_poly(__dmul_rn(t, t)));
    } else {
        om = 2.0 * atan2(im, re);
    }
    if constexpr (kPhi) phi = __fma_rn(-Y, om, sphi);
    if constexpr (kField) {
        Ex = sx;
        Ey = om;
        Ez = sz;
    }
}

// Element e and its edges seen from the local point (X, Y, Z).
template <bool kPhi, bool kField>
__device__ __forceinline__ void elem_at_f64(const Elem& e, const PolyEdges& g, double X, double Y, double Z,
                                            double& phi, double& lx, double& ly, double& lz) {
    if (e.nv == 4)
        poly_f64<4, kPhi, kField>(e, g, X, Y, Z, phi, lx, ly, lz);
    else
        poly_f64<3, kPhi, kField>(e, g, X, Y, Z, phi, lx, ly, lz);
}

// Local coordinates of the global vector (dx, dy, dz).
__device__ __forceinline__ void to_local(const Elem& e, double dx, double dy, double dz, double& X, double& Y,
                                         double& Z) {
    X = __fma_rn(dx, e.ex[0], __fma_rn(dy, e.ex[1], __dmul_rn(dz, e.ex[2])));
    Y = __fma_rn(dx, e.ey[0], __fma_rn(dy, e.ey[1], __dmul_rn(dz, e.ey[2])));
    Z = __fma_rn(dx, e.ez[0], __fma_rn(dy, e.ez[1], __dmul_rn(dz, e.ez[2])));
}

// Local influence of element e at a global point (Px, Py, Pz) by the general form (the near
// pairs of the mixed paths, single elements); self forces Y = 0.
__device__ __forceinline__ void elem_local_f64(const Elem& e, double Px, double Py, double Pz, bool self,
                                               double& phi, double& lx, double& ly, double& lz) {
    double X, Y, Z;
    to_local(e, __dsub_rn(Px, e.o[0]), __dsub_rn(Py, e.o[1]), __dsub_rn(Pz, e.o[2]), X, Y, Z);
    if (self) Y = 0.0;
    if (e.nv == 4)
        poly_general<4>(e, X, Y, Z, phi, lx, ly, lz);
    else
        poly_general<3>(e, X, Y, Z, phi, lx, ly, lz);
}

// A tile of kTile64 elements for the FP64 sums over (element, image) pairs, in shared memory:
// element records, edges, and tau_k = t_k in the element's frame, so that a pair's local
// coordinates are X0 - tau_k (three operations; X0 = (P - o) in the frame, once per element and
// point) instead of a difference and a rotation per pair.
constexpr int kTile64 = 8;
struct Tile64 {
    Elem el[kTile64];
    PolyEdges edge[kTile64];
    double tau[kTile64][kMaxImg][3];
};
// Loads the elements [base, base + cnt); called by every thread of the block, with a barrier on
// both sides.
__device__ __forceinline__ void load_tile64(Tile64& s, const Elem* __restrict__ el, int64_t base, int cnt,
                                            const ImageTable& img) {
    __syncthreads();
    const double2* src = reinterpret_cast<const double2*>(el + base);
    double2* dst = reinterpret_cast<double2*>(s.el);
    for (int i = threadIdx.x; i < cnt * 16; i += blockDim.x) dst[i] = src[i];
    __syncthreads();
    for (int i = threadIdx.x; i < cnt * 4; i += blockDim.x)
        if (i % 4 < s.el[i / 4].nv) poly_edge(s.el[i / 4], i % 4, s.edge[i / 4]);
    for (int i = threadIdx.x; i < cnt * img.n; i += blockDim.x) {
        const int jj = i / img.n, k = i - jj * img.n;
        to_local(s.el[jj], img.t[k][0], img.t[k][1], img.t[k][2], s.tau[jj][k][0], s.tau[jj][k][1], s.tau[jj][k][2]);
    }
    __syncthreads();
}

}  // namespace nb
