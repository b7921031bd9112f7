// fill_mixed.cu -- mixed-precision influence-matrix fill (Eq. Matrix, collocation at
// centroids, periodic images):
//   conductor row i:  K_ij = ke sum_k Phi'(c_i - t_k; j)
//   interface row i:  K_ij = ke sum_k n_i . E'(c_i - t_k; j) + delta_ij diag_i
//
// Far pairs (distance to the image centroid >= kFillRatioC element radii) are evaluated in two-float
// arithmetic: every quantity is an unevaluated sum hi + lo of two FP32 values and products and
// sums keep their rounding errors through error-free transformations (Dekker / Knuth TwoSum,
// FMA-based TwoProd), about 44 significant bits.  From 32 radii on (interface rows: 52) a pair
// is the element's moments (fill_mom_phi2, fill_mom_field2 of twofloat.cuh), two images per packed
// FP32x2 instruction; nearer, one to three pairs in a hundred, Gauss rules whose truncation stays
// below ~3e-12 of the pair (tiers in nb_internal.h).  Near pairs use the FP64 closed forms of
// influence.cuh.  The FP32 pipe runs 64 times the FP64 rate on this GPU, so a pair by moments (201
// or 427 FP32 lane operations) costs as much as three to seven FP64 operations.
//
// Geometry of one pair in the local frame of the column element j (origin anywhere, axes
// ex, ey = normal, ez): D = c_i - (c_j + t_k) has components
//   X = (c_i - c_j) . ex - t_k . ex,  Y, Z likewise,
// the first term once per (i, j), the second (tau) tabulated per (j, k).  A node at
// offset s = centroid - node (in the element plane, local (s_x, s_z)) sees the target at
// P - node = D + s, so
//   r^2 = |D|^2 + q,  q = 2 (X s_x + Z s_z) + |s|^2,
// which needs only two products per node.  1/r comes from one MUFU rsqrt refined by one
// Newton step carried in two-float form; Phi' += w / r, n . E' += w (n . (D + s)) / r^3.
//
// Kernel k_fill_far: thread per row i, grid.y over column chunks; column tiles (element
// records, moments, tau) staged in shared memory.  It writes
// ke * (far sum) (+ the interface diagonal) to every entry.  Kernel k_fill_near: warp
// per row i; it visits the image centroids in the 27 grid cells around c_i (cell edge >=
// the largest near radius) and adds ke * (FP64 closed form) of every near pair.  Both
// decide "near" by the same rounded FP32 squared distance (pair_d2 of eval_blocks.cuh) on
// the same two-float inputs, so every pair is counted exactly once.
#include "twofloat.cuh"

namespace nb {

namespace {

constexpr int kFT = 128;       // threads per block (one row each)
constexpr int kFillBlocks = 4;  // resident far blocks per SM

// Phi' nodes: S += w / r (sh = hi sum, nl = -lo sum), two nodes per step
__device__ __forceinline__ void nodes_phi2(const float4* __restrict__ nd, int pairs, const PairDF2& P, float2& sh,
                                           float2& nl) {
    const float2 m1 = bc2(-1.f);
    for (int q = 0; q < pairs; ++q) {
        const float4 q0 = nd[4 * q], q1 = nd[4 * q + 1], q2 = nd[4 * q + 2], q3 = nd[4 * q + 3];
        float2 y0, ny0, nyl, a, na, nae;
        node_rinv2(P, q0, q1, q2, q3, y0, ny0, nyl, a, na, nae);
        const float2 w = make_float2(q1.z, q1.w), wl = make_float2(q3.z, q3.w);
        const float2 m = __fmul2_rn(w, y0);
        float2 nme = __ffma2_rn(w, ny0, m);  // m - w y0
        nme = __ffma2_rn(w, nyl, nme);
        nme = __ffma2_rn(wl, ny0, nme);
        float2 t;
        two_sum2(sh, m, sh, t);
        nl = __ffma2_rn(t, m1, __fadd2_rn(nl, nme));
    }
}

// n . E' nodes: S += w (n . (D + s)) / r^3, with n . s = (n . ex) s_x + (n . ez) s_z
__device__ __forceinline__ void nodes_nE2(const float4* __restrict__ nd, int pairs, const PairDF2& P,
                                          const NormDF2& Nn, float2& sh, float2& nl) {
    const float2 m1 = bc2(-1.f), half = bc2(0.5f);
    for (int q = 0; q < pairs; ++q) {
        const float4 q0 = nd[4 * q], q1 = nd[4 * q + 1], q2 = nd[4 * q + 2], q3 = nd[4 * q + 3];
        float2 y0, ny0, nyl, a, na, nae;
        node_rinv2(P, q0, q1, q2, q3, y0, ny0, nyl, a, na, nae);
        const float2 sx = make_float2(q0.x, q0.y), sz = make_float2(q0.z, q0.w);
        const float2 sxl = make_float2(q2.x, q2.y), szl = make_float2(q2.z, q2.w);
        // 2 (n . s)
        const float2 p1 = __fmul2_rn(Nn.nxh, sx), ne1 = __ffma2_rn(Nn.nnxh, sx, p1);
        const float2 p2 = __fmul2_rn(Nn.nzh, sz), ne2 = __ffma2_rn(Nn.nnzh, sz, p2);
        float2 ns, t;
        two_sum2(p1, p2, ns, t);
        float2 nsl = __ffma2_rn(ne1, m1, t);
        nsl = __ffma2_rn(ne2, m1, nsl);
        nsl = __ffma2_rn(Nn.nxh, sxl, nsl);
        nsl = __ffma2_rn(Nn.nxl, sx, nsl);
        nsl = __ffma2_rn(Nn.nzh, szl, nsl);
        nsl = __ffma2_rn(Nn.nzl, sz, nsl);
        // g = n . (D + s)
        float2 gh, t2;
        two_sum2(Nn.ndh, __fmul2_rn(half, ns), gh, t2);
        const float2 gl = __fadd2_rn(__ffma2_rn(half, nsl, Nn.ndl), t2);
        // y^3 = y^2 y, y^2 = a + (ae + 2 y0 yl): negated low parts
        const float2 ny2l = __ffma2_rn(__fadd2_rn(y0, y0), nyl, nae);
        const float2 c3 = __fmul2_rn(a, y0);
        float2 nc3e = __ffma2_rn(na, y0, c3);  // c3 - a y0
        nc3e = __ffma2_rn(a, nyl, nc3e);
        nc3e = __ffma2_rn(ny2l, y0, nc3e);
        // w y^3 = m + me
        const float2 w = make_float2(q1.z, q1.w), wl = make_float2(q3.z, q3.w);
        const float2 nc3 = __fmul2_rn(c3, m1);
        const float2 m = __fmul2_rn(w, c3);
        float2 nme = __ffma2_rn(w, nc3, m);  // m - w c3
        nme = __ffma2_rn(w, nc3e, nme);
        nme = __ffma2_rn(wl, nc3, nme);
        // (w y^3) g = f + fe
        const float2 nm = __fmul2_rn(m, m1);
        const float2 f = __fmul2_rn(m, gh);
        float2 nfe = __ffma2_rn(nm, gh, f);  // f - m gh
        nfe = __ffma2_rn(nm, gl, nfe);
        nfe = __ffma2_rn(nme, gh, nfe);
        float2 t3;
        two_sum2(sh, f, sh, t3);
        nl = __ffma2_rn(t3, m1, __fadd2_rn(nl, nfe));
    }
}

__device__ __forceinline__ void stage(float4* dst, const float4* __restrict__ src, int cnt) {
    for (int i = threadIdx.x; i < cnt; i += blockDim.x) dst[i] = src[i];
}

// Dynamic shared memory per tile of te elements: FillEl (9 float4), FillMom, and tau as six planes of
// nimg (padded to even) floats (x, y, z negated: hi, then lo).
__host__ __device__ constexpr int fill_pad(int nimg) { return (nimg + 1) & ~1; }
__host__ __device__ constexpr int fill_tile_f4(int te, int nimg) {
    return te * (9 + kFillMomF4) + (te * 6 * fill_pad(nimg) + 3) / 4;
}

// The pair (row i, element j, image k) by its tier's nodes where it is nearer than the moments reach (one
// to three pairs in a hundred); a near pair is left to k_fill_near.
__device__ __noinline__ void fill_pair_nodes(const float4* __restrict__ nd, const float4* __restrict__ cjk2,
                                             const float4& hdr, const float (&ch)[3], const float (&cl)[3],
                                             const float (&Xh)[3], const float (&Xl)[3], bool iface, const FillRow& R,
                                             float2& sh, float2& snl) {
    float dx, dy, dz;
    if (!(pair_d2(ch[0], ch[1], ch[2], cl[0], cl[1], cl[2], cjk2[0], cjk2[1], dx, dy, dz) >= hdr.z)) return;
    float d2h, d2l;
    df_norm2(Xh[0], Xl[0], Xh[1], Xl[1], Xh[2], Xl[2], d2h, d2l);
    PairDF2 P;
    P.xh = bc2(Xh[0]), P.nxh = bc2(-Xh[0]), P.xl = bc2(Xl[0]);
    P.zh = bc2(Xh[2]), P.nzh = bc2(-Xh[2]), P.zl = bc2(Xl[2]);
    P.d2h = bc2(d2h), P.d2l = bc2(d2l);
    if (!iface) {
        nodes_phi2(nd + kFillOffC, kFillPairsC, P, sh, snl);
        return;
    }
    NormDF2 Nn;
    Nn.nxh = bc2(R.nxh), Nn.nnxh = bc2(-R.nxh), Nn.nxl = bc2(R.nxl);
    Nn.nzh = bc2(R.nzh), Nn.nnzh = bc2(-R.nzh), Nn.nzl = bc2(R.nzl);
    float ndh, ndl;
    df_dot3(Xh, Xl, make_float4(R.nxh, R.nyh, R.nzh, 0.f), make_float4(R.nxl, R.nyl, R.nzl, 0.f), ndh, ndl);
    Nn.ndh = bc2(ndh), Nn.ndl = bc2(ndl);
    const bool b = d2h >= hdr.y;
    nodes_nE2(nd + (b ? kFillOffB : kFillOffC), b ? kFillPairsB : kFillPairsC, P, Nn, sh, snl);
}

// Far pairs of a block's 128 rows and `cols` columns: the moments from 32 radii on (interface rows:
// 52), nodes nearer.  9,996 elements x 25 copies (18 % interface rows) took 71 ms with nodes
// for every pair and 35 ms so; bound by the FP32 pipe.
__global__ void __launch_bounds__(kFT, kFillBlocks)
    k_fill_far(const FillEl* __restrict__ fe, const float4* __restrict__ nodes, const float4* __restrict__ mom,
               const float4* __restrict__ tau, const float4* __restrict__ cjk, const double* __restrict__ diag_in,
               int64_t n, int nimg, int te, int cols, double* __restrict__ K) {
    extern __shared__ float4 sm[];
    FillEl* s_fe = reinterpret_cast<FillEl*>(sm);
    float4* s_mom = sm + 9 * te;
    float* s_tau = reinterpret_cast<float*>(s_mom + kFillMomF4 * te);
    const int np2 = fill_pad(nimg);

    const int64_t i = (int64_t)blockIdx.x * kFT + threadIdx.x;
    const bool active = i < n;
    // row data: centroid and normal (two floats each), row type
    float ch[3] = {0.f, 0.f, 0.f}, cl[3] = {0.f, 0.f, 0.f}, nh[3] = {0.f, 0.f, 0.f}, nl[3] = {0.f, 0.f, 0.f};
    bool iface = false;
    double diag = 0.0;
    if (active) {
        const FillEl r = fe[i];
        ch[0] = r.ch.x, ch[1] = r.ch.y, ch[2] = r.ch.z;
        cl[0] = r.cl.x, cl[1] = r.cl.y, cl[2] = r.cl.z;
        nh[0] = r.eyh.x, nh[1] = r.eyh.y, nh[2] = r.eyh.z;
        nl[0] = r.eyl.x, nl[1] = r.eyl.y, nl[2] = r.eyl.z;
        diag = diag_in[i];
        iface = diag != 0.0;  // interface rows carry the nonzero diagonal term
    }
    const double ke = 1.0 / (4.0 * kPi * kEps0);
    const int64_t j0 = (int64_t)blockIdx.y * cols;
    const int64_t j1 = min(n, j0 + cols);
    for (int64_t base = j0; base < j1; base += te) {
        const int cnt = (int)min((int64_t)te, j1 - base);
        __syncthreads();
        stage(reinterpret_cast<float4*>(s_fe), reinterpret_cast<const float4*>(fe + base), 9 * cnt);
        stage(s_mom, mom + base * kFillMomF4, kFillMomF4 * cnt);
        for (int q = threadIdx.x; q < cnt * np2; q += blockDim.x) {
            const int jj = q / np2, k = min(q - jj * np2, nimg - 1);
            const float4 h = tau[2 * ((base + jj) * nimg + k)], l = tau[2 * ((base + jj) * nimg + k) + 1];
            float* d = s_tau + jj * 6 * np2 + (q - jj * np2);
            d[0] = -h.x, d[np2] = -h.y, d[2 * np2] = -h.z;
            d[3 * np2] = -l.x, d[4 * np2] = -l.y, d[5 * np2] = -l.z;
        }
        __syncthreads();
        for (int jj = 0; jj < cnt; ++jj) {
            const FillEl& E = s_fe[jj];
            const float4* M = s_mom + kFillMomF4 * jj;
            const int64_t j = base + jj;
            const float* nt = s_tau + jj * 6 * np2;
            // c_i - c_j and its local components
            float dh[3], dl[3];
            df_sub(ch[0], cl[0], E.ch.x, E.cl.x, dh[0], dl[0]);
            df_sub(ch[1], cl[1], E.ch.y, E.cl.y, dh[1], dl[1]);
            df_sub(ch[2], cl[2], E.ch.z, E.cl.z, dh[2], dl[2]);
            float x0h, x0l, y0h, y0l, z0h, z0l;
            df_dot3(dh, dl, E.exh, E.exl, x0h, x0l);
            df_dot3(dh, dl, E.eyh, E.eyl, y0h, y0l);
            df_dot3(dh, dl, E.ezh, E.ezl, z0h, z0l);
            FillRow R;
            if (iface) {
                df_dot3(nh, nl, E.exh, E.exl, R.nxh, R.nxl);
                df_dot3(nh, nl, E.eyh, E.eyl, R.nyh, R.nyl);
                df_dot3(nh, nl, E.ezh, E.ezl, R.nzh, R.nzl);
                // gx = 2 a1 n_x + a2 n_z, gz = a2 n_x + 2 a3 n_z
                auto dot2 = [](float ah, float al, float bh, float bl, float xh, float xl, float zh, float zl, float& h,
                               float& l) {
                    float p, e, q, f, t;
                    two_prod(ah, xh, p, e);
                    two_prod(bh, zh, q, f);
                    two_sum(p, q, h, t);
                    e = __fmaf_rn(ah, xl, __fmaf_rn(al, xh, e));
                    f = __fmaf_rn(bh, zl, __fmaf_rn(bl, zh, f));
                    l = __fadd_rn(t, __fadd_rn(e, f));
                };
                dot2(M[0].x + M[0].x, M[0].z + M[0].z, M[1].x, M[1].z, R.nxh, R.nxl, R.nzh, R.nzl, R.gxh, R.gxl);
                dot2(M[1].x, M[1].z, M[2].x + M[2].x, M[2].z + M[2].z, R.nxh, R.nxl, R.nzh, R.nzl, R.gzh, R.gzl);
            }
            float2 sh = bc2(0.f), snl = bc2(0.f);  // node sums: hi, negated lo
            float2 Sh = bc2(0.f), Sl = bc2(0.f);   // moment sums
            const float mom2 = iface ? E.hdr.y * (float)(kFillMomField * kFillMomField / (kFillRatioB * kFillRatioB))
                                     : E.hdr.y;
            uint32_t nearer = 0;  // images of the group of 32 at hand that the moments do not reach
            for (int k = 0; k < np2; k += 2) {
                auto diff = [&](float ah, float al, int q, float2& h, float2& l) {
                    float2 t;
                    two_sum2(bc2(ah), *reinterpret_cast<const float2*>(nt + q * np2 + k), h, t);
                    l = __fadd2_rn(t, __fadd2_rn(bc2(al), *reinterpret_cast<const float2*>(nt + (q + 3) * np2 + k)));
                };
                auto square = [](float2 h, float2 l, float2& p, float2& e) {
                    p = __fmul2_rn(h, h);
                    e = __ffma2_rn(__fadd2_rn(h, h), l, __ffma2_rn(h, h, make_float2(-p.x, -p.y)));
                };
                FillPair2 P;
                float2 yh, yl, py, ey, s, t1, t2;
                diff(x0h, x0l, 0, P.xh, P.xl);
                diff(y0h, y0l, 1, yh, yl);
                diff(z0h, z0l, 2, P.zh, P.zl);
                square(P.xh, P.xl, P.px, P.ex);
                square(yh, yl, py, ey);
                square(P.zh, P.zl, P.pz, P.ez);
                two_sum2(P.px, py, s, t1);
                two_sum2(s, P.pz, P.d2h, t2);
                P.d2l = __fadd2_rn(__fadd2_rn(P.ex, ey), __fadd2_rn(P.ez, __fadd2_rn(t1, t2)));
                const bool two = k + 1 < nimg;
                const bool far0 = P.d2h.x >= mom2, far1 = two && P.d2h.y >= mom2;
                if (iface)
                    fill_mom_field2(M, R, P, yh, yl, far0, far1, Sh, Sl);
                else
                    fill_mom_phi2(M, P, far0, far1, Sh, Sl);
                nearer |= ((far0 ? 0u : 1u) | (far1 || !two ? 0u : 2u)) << (k & 31);
                if ((k & 31) == 30 || k + 2 >= np2) {
                    for (uint32_t m = nearer; m; m &= m - 1) {
                        const int kk = (k & ~31) + __ffs(m) - 1;
                        float Xh[3], Xl[3];
                        df_sub(x0h, x0l, -nt[kk], -nt[3 * np2 + kk], Xh[0], Xl[0]);
                        df_sub(y0h, y0l, -nt[np2 + kk], -nt[4 * np2 + kk], Xh[1], Xl[1]);
                        df_sub(z0h, z0l, -nt[2 * np2 + kk], -nt[5 * np2 + kk], Xh[2], Xl[2]);
                        fill_pair_nodes(nodes + j * kFillNodeRec, cjk + 2 * (j * nimg + kk), E.hdr, ch, cl, Xh, Xl,
                                        iface, R, sh, snl);
                    }
                    nearer = 0;
                }
            }
            if (active) {
                // A (sum over the images) in two floats; the node sums' lanes (hi + lo each) in FP64
                const float4 area = M[kFillMomF4 - 1];
                float h, t, p, e;
                two_sum(Sh.x, Sh.y, h, t);
                const float l = __fadd_rn(t, __fadd_rn(Sl.x, Sl.y));
                two_prod(h, area.x, p, e);
                e = __fmaf_rn(h, area.y, __fmaf_rn(l, area.x, e));
                const double acc =
                    ((double)p + (double)e) + (((double)sh.x - (double)snl.x) + ((double)sh.y - (double)snl.y));
                K[i + j * n] = (i == j) ? fma(ke, acc, diag) : ke * acc;
            }
        }
    }
}

// FillMom records (twofloat.cuh) from the elements' 36-node rules, which integrate degree 6 exactly:
//   |u|^l P_l(cos(D, u)) = sum_m c_lm (D.u / d)^(l - 2m) |u|^2m,  c_lm = (-1)^m (2l - 2m)! / (2^l m! (l-m)! (l-2m)!).
__global__ void k_fill_moments(const FillEl* __restrict__ fe, const float4* __restrict__ nodes, int64_t n,
                               float4* __restrict__ mom) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const double s = exp2(ceil(log2((double)fe[j].ch.w)));
    const float4* nd = nodes + j * kFillNodeRec + kFillOffC;
    double M[7][7];  // moments of ((node - centroid) / s)_x^a (..)_z^b, over A below
    for (int a = 0; a < 7; ++a)
        for (int b = 0; b < 7; ++b) M[a][b] = 0.0;
    for (int q = 0; q < 2 * kFillPairsC; ++q) {
        const float4* r = nd + 4 * (q / 2);
        const bool o = q & 1;
        const double x = -0.5 / s * (o ? (double)r[0].y + (double)r[2].y : (double)r[0].x + (double)r[2].x);
        const double z = -0.5 / s * (o ? (double)r[0].w + (double)r[2].w : (double)r[0].z + (double)r[2].z);
        double px = o ? (double)r[1].w + (double)r[3].w : (double)r[1].z + (double)r[3].z;  // w x^a z^b
        for (int a = 0; a < 7; ++a, px *= x) {
            double v = px;
            for (int b = 0; a + b < 7; ++b, v *= z) M[a][b] += v;
        }
    }
    const double A = M[0][0];
    const double fact[13] = {1, 1, 2, 6, 24, 120, 720, 5040, 40320, 362880, 3628800, 39916800, 479001600};
    double c[8 + kFillMomCoef + 1];
    const double quad[4] = {1.5 * M[2][0] / A, 3.0 * M[1][1] / A, 1.5 * M[0][2] / A, -0.5 * (M[2][0] + M[0][2]) / A};
    for (int q = 0; q < 4; ++q) {
        c[2 * q] = quad[q];
        c[2 * q + 1] = quad[q] - (double)__double2float_rn(quad[q]);
    }
    for (int i = 0; i < 7; ++i)
        for (int k = i; k < 7; ++k)
            for (int t = 0; t < fill_mom_terms(k); ++t) {
                const int jz = k - i, m = fill_mom_m0(k) + t, l = k + 2 * m;
                double v = 0.0;  // integral of u_x^i u_z^jz |u|^2m
                for (int r = 0; r <= m; ++r)
                    v += fact[m] / (fact[r] * fact[m - r]) * M[i + 2 * r][jz + 2 * (m - r)];
                const double clm = (m & 1 ? -1.0 : 1.0) * fact[2 * l - 2 * m] /
                                   ((double)(1 << l) * fact[m] * fact[l - m] * fact[k]);
                c[8 + fill_mom_off(i, jz) + t] = clm * fact[k] / (fact[i] * fact[jz]) * v / A;
            }
    c[8 + kFillMomCoef] = 0.0;
    float4* out = mom + j * kFillMomF4;
    for (int q = 0; q < kFillMomF4 - 1; ++q) {
        const float a = (float)c[2 * q], b = (float)c[2 * q + 1];
        out[q] = make_float4(a, a, b, b);
    }
    const float ah = (float)A;
    out[kFillMomF4 - 1] = make_float4(ah, (float)(A - (double)ah), (float)s, (float)(s * s));
}

// Near pairs of row i by one warp: found and queued 32 at a time as in near_point_warp, evaluated 32 at a
// time (an FP64 instruction holds the pipe as long for one lane as for 32).  Two near copies of one
// column meet in the same entry: a batch that holds such a pair adds its values lane by lane, so
// the order is fixed.  9,996 elements x 25 copies, 238 near pairs a row: 17.8 ms with a thread per row,
// 2.0 ms so.
__global__ void __launch_bounds__(128) k_fill_near(const Elem* __restrict__ el, const FillEl* __restrict__ fe,
                                                   const float4* __restrict__ cjk, int64_t n, const ImageTable img,
                                                   const NearGrid grid, const int32_t* __restrict__ cell_start,
                                                   const int32_t* __restrict__ cell_items, double* __restrict__ K) {
    __shared__ int32_t s_queue[4][kNearQueue];
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= n) return;
    const Elem& ei = el[i];
    const double Px = ei.c[0], Py = ei.c[1], Pz = ei.c[2];
    const double nx = ei.ey[0], ny = ei.ey[1], nz = ei.ey[2];
    const bool cond = ei.bc == NEBEM_CONDUCTOR;
    const float4 rh = fe[i].ch, rl = fe[i].cl;
    const int nimg = img.n;
    const double ke = 1.0 / (4.0 * kPi * kEps0);
    near_pairs_warp(
        Px, Py, Pz, rh.x, rh.y, rh.z, rl.x, rl.y, rl.z, cjk, grid, cell_start, cell_items, nimg, NearFill{fe},
        s_queue[threadIdx.x >> 5], [&](bool live, int32_t jk) {
            const int32_t j = jk / nimg, k = jk - j * nimg;
            double v = 0.0;
            if (live) {
                const Elem& e = el[j];
                const bool self = (i == j) && (k == img.k0);
                double f, gx, gy, gz;
                elem_local_f64(e, Px - img.t[k][0], Py - img.t[k][1], Pz - img.t[k][2], self, f, gx, gy, gz);
                if (cond) {
                    v = f;
                } else {
                    const double Ex = __fma_rn(gx, e.ex[0], __fma_rn(gy, e.ey[0], __dmul_rn(gz, e.ez[0])));
                    const double Ey = __fma_rn(gx, e.ex[1], __fma_rn(gy, e.ey[1], __dmul_rn(gz, e.ez[1])));
                    const double Ez = __fma_rn(gx, e.ex[2], __fma_rn(gy, e.ey[2], __dmul_rn(gz, e.ez[2])));
                    v = __fma_rn(nx, Ex, __fma_rn(ny, Ey, __dmul_rn(nz, Ez)));
                }
            }
            double* at = K + i + (int64_t)j * n;
            const unsigned same = __match_any_sync(0xffffffffu, live ? j : -1 - (int)(threadIdx.x & 31));
            if (__any_sync(0xffffffffu, __popc(same) > 1)) {
                for (int l = 0; l < 32; ++l) {
                    if (live && (int)(threadIdx.x & 31) == l) *at = __fma_rn(ke, v, *at);
                    __syncwarp();
                }
            } else if (live) {
                *at = __fma_rn(ke, v, *at);
            }
        });
}

}  // namespace

size_t fill_moments_bytes(int64_t n) { return sizeof(float4) * kFillMomF4 * (size_t)n; }
cudaError_t launch_fill_moments(const FillEl* fe, const float4* nodes, int64_t n, float4* mom, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_fill_moments<<<(unsigned)((n + 31) / 32), 32, 0, s>>>(fe, nodes, n, mom);
    return cudaGetLastError();
}

cudaError_t launch_fill_mixed(const Elem* el, const FillEl* fe, const float4* nodes, const float4* mom,
                              const float4* tau, const float4* cjk, const double* diag, int64_t n,
                              const ImageTable& img, const NearGrid& grid, const int32_t* cell_start,
                              const int32_t* cell_items, double* K, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    // column tile: as many elements as fit in ~40 KB (four blocks per SM), at most 16
    constexpr int kSmem = 40 * 1024;
    int te = 16;
    while (te > 1 && fill_tile_f4(te, img.n) * (int)sizeof(float4) > kSmem) --te;
    const size_t smem = (size_t)fill_tile_f4(te, img.n) * sizeof(float4);
    // one value whatever the tile: another thread's call may be between this and its launch
    cudaError_t e = cudaFuncSetAttribute(k_fill_far, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    if (e != cudaSuccess) return e;
    int cols = 0;
    e = fill_cols(n, kFT, kFillBlocks, &cols);
    if (e != cudaSuccess) return e;
    dim3 g1((unsigned)((n + kFT - 1) / kFT), (unsigned)((n + cols - 1) / cols));
    k_fill_far<<<g1, kFT, smem, s>>>(fe, nodes, mom, tau, cjk, diag, n, img.n, te, cols, K);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_fill_near<<<(unsigned)((n + 3) / 4), 128, 0, s>>>(el, fe, cjk, n, img, grid, cell_start, cell_items, K);
    return cudaGetLastError();
}

}  // namespace nb
