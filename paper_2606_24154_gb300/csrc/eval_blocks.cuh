// eval_blocks.cuh -- per-block evaluation bodies shared by the standalone evaluation
// kernels (eval_f64.cu, eval_mixed.cu) and the serving kernel (server.cu): one thread per
// target, `count` <= blockDim.x targets starting at `pts`.  Using the same functions in
// both places makes a point's result identical whichever launch evaluates it.
//
// Mixed precision.
//
// Same sums as the FP64 kernel (Eq. Potential / Eq. Field over elements and periodic
// images), but each (point, element, image) pair picks its arithmetic by its distance d
// to the image centroid, in units of the element's circumradius rho:
//   d >= ratio_0 rho      FP32 Gauss rule, tier 0 (4 nodes)
//   d >= ratio_a rho      FP32 Gauss rule, tier a (6 nodes triangle / 9 rectangle)
//   d >= ratio_b rho      FP32 Gauss rule, tier b (16 nodes)
//   d >= ratio_near rho   FP32 Gauss rule, tier c (36 nodes)
//   nearer                FP64 closed form (influence.cuh), where ln/atan cancel
// Quadrature per node: Phi += w / r, E += w (P - x_n) / r^3 with one rsqrt; two nodes at
// a time in the packed FP32x2 instructions (half the issue slots of scalar FP32).
//
// Two kernels: k_eval_far runs every FP32 tier over all (element, image) pairs and skips
// near pairs; k_eval_near visits only the image centroids in the 27 grid cells around
// each point (a cell list built per geometry, cell edge >= the largest near radius) and
// adds the near pairs' FP64 closed forms.  Keeping the FP64 code out of the far kernel
// keeps its register count (and so its occupancy) at the FP32 kernel's level.  Both
// kernels decide "near" with the same rounded FP32 operations (pair_d2) on the same
// inputs, so every pair is counted exactly once.
//
// The FP32 difference P - x_n keeps its relative accuracy even when P and the node are
// millimetres from the origin but micrometres apart: both sides are held as two floats
// (hi + lo) and (P_hi - C_hi) + (P_lo - C_lo) is formed first, C = c_j + t_k being the
// image centroid (FP64 sum split once per geometry).  Node offsets from the centroid are
// small, so the remaining FP32 operations carry ~1e-7 relative error.
//
// Accumulation: per element over its images in FP32, weighted by sigma_j, summed in FP32
// over groups of kGroup elements and flushed to FP64.  Every decision depends only on the
// pair, and each point's sums run in a fixed order, so a point's result is bit-identical
// whatever other points share its launch.
//
// Error scales.  Beside the sums, the far part accumulates per point the scales of its
// rounding and truncation errors from the per-element terms b_j = |sigma_j| |sum_k Phi'_jk|
// (for E: |sigma_j| |sum_k E'_jk|_1) over the FP32 pairs: their sum B = sum_j b_j and their
// root sum of squares S = sqrt(sum_j b_j^2).  Errors that keep their sign from element to
// element (the Gauss rules' truncation) grow with B; rounding errors, whose signs vary
// from element to element, add up like a random sum and grow with S, which is far smaller
// than B when many elements contribute alike.  eval_acc.cu turns the scales into a
// per-point error estimate and refines the points whose estimate exceeds the requested
// relative tolerance.  The scales do not enter the sums themselves.
#pragma once
#include "influence.cuh"

namespace nb {

constexpr int kEvalThreads = 128;  // threads per block (one target each)
constexpr int kTileMax = 16;       // elements per shared-memory tile (mixed)
constexpr int kCjkMax = 512;       // (element, image) centres per tile (mixed)
constexpr int kGroup = 8;          // elements per FP32 partial sum (mixed)

// Summation tree over the elements, the same in every launch: leaves of kLeafEl elements
// (a multiple of every tile width), added in order to chunks of kChunkEl, added in order to
// the total.  A launch may take a point's whole sum, or its chunks or its leaves as separate
// pieces on different blocks (SplitPlan); the tree, and so every bit, stays the same.
constexpr int kLeafEl = 32;
constexpr int kChunkEl = 256;
static_assert(kChunkEl % kLeafEl == 0 && kLeafEl % kTileMax == 0 && kLeafEl % kTile64 == 0, "summation tree");

// How G groups of kEvalThreads points are dealt to the gb blocks that the device holds at once:
// the first Gm groups whole, floor(G / gb) - 1 rounds of gb; the R < 2 gb left over in R * np
// pieces (group, chunk), or (group, leaf) where the chunks would give a block fewer than
// kSplitRounds pieces.  (With the last full round whole too, its slowest groups ran on alone:
// 169 ms instead of 144 for the FP32 pass over 233,472 points, exactly two rounds.)  One thread walks all
// (element, image) pairs of its point in turn, about 0.29 us a pair whatever else the SM does, so a launch cannot end before its longest piece:
// 250,000 pairs (72 ms) for a whole point of a 10,000-element cell with 25 copies, 1.9 ms for a
// chunk, 0.23 ms for a leaf.  The leaves cost eight times the chunks' partial sums (48 B per
// point and piece), which is why they are kept for launches that are short of pieces.  Where the pieces' sums
// do not fit in the `cap` sums that the caller has room for, more groups are taken whole: the same bits, with a
// longer last round.
constexpr int kSplitRounds = 4;
struct SplitPlan {
    int64_t Gm, R, np;
    int leaf;  // 1: pieces are leaves, 0: chunks
};
// pieces of `len` elements (at least one: an empty set has one empty piece)
__host__ __device__ __forceinline__ int64_t split_count(int64_t n_el, int64_t len) {
    return n_el > 0 ? (n_el + len - 1) / len : 1;
}
__host__ __device__ __forceinline__ SplitPlan split_plan(int64_t G, int64_t gb, int64_t n_el, int64_t cap) {
    SplitPlan s;
    s.Gm = G >= 2 * gb ? (G / gb - 1) * gb : 0;
    s.R = G - s.Gm;
    const int64_t nch = split_count(n_el, kChunkEl), nleaf = split_count(n_el, kLeafEl);
    s.leaf = s.R * nch < kSplitRounds * gb && s.R * nleaf * kEvalThreads <= cap;
    s.np = s.leaf ? nleaf : nch;
    if (s.R * s.np * kEvalThreads > cap) {
        s.R = cap / (s.np * kEvalThreads);
        s.Gm = G - s.R;
    }
    return s;
}
// partial sums (one per point and piece) of the largest left-over part of up to G groups
inline int64_t split_parts(int64_t G, int64_t gb, int64_t n_el) {
    const int64_t nch = split_count(n_el, kChunkEl), nleaf = split_count(n_el, kLeafEl);
    const int64_t r = G < 2 * gb ? G : 2 * gb;                      // groups left over, at most
    const int64_t rl = (kSplitRounds * gb + nch - 1) / nch;          // the most that go by leaves
    const int64_t a = r * nch, b = (r < rl ? r : rl) * nleaf;
    return (a > b ? a : b) * kEvalThreads;
}
// bytes of that many sums of type T, at most kPartMax
template <class T>
inline size_t split_part_bytes(int64_t npts, int64_t gb, int64_t n_el) {
    const size_t b = sizeof(T) * (size_t)split_parts((npts + kEvalThreads - 1) / kEvalThreads, gb, n_el);
    return b < kPartMax ? b : kPartMax;
}
// The piece that unit u (< Gm + R np) stands for: its group and element range.
struct SplitUnit {
    int64_t group, e0, e1, r, piece;
    bool whole;
};
__device__ __forceinline__ SplitUnit split_unit(const SplitPlan& s, int64_t u, int64_t n_el) {
    SplitUnit t;
    t.whole = u < s.Gm;
    if (t.whole) {
        t.group = u, t.e0 = 0, t.e1 = n_el, t.r = 0, t.piece = 0;
        return t;
    }
    // consecutive units: the same piece of other groups, whose element data then stay in L2
    t.piece = (u - s.Gm) / s.R;
    t.r = (u - s.Gm) - t.piece * s.R;
    t.group = s.Gm + t.r;
    const int64_t len = s.leaf ? kLeafEl : kChunkEl;
    t.e0 = t.piece * len;
    t.e1 = t.e0 + len < n_el ? t.e0 + len : n_el;
    return t;
}

// Squared FP32 distance between a point (two floats per coordinate) and an image centroid;
// the operation sequence is pinned (no contraction) so both kernels agree bit for bit.
__device__ __forceinline__ float pair_d2(float phx, float phy, float phz, float plx, float ply, float plz,
                                         const float4& ch, const float4& cl, float& dx, float& dy, float& dz) {
    dx = __fadd_rn(__fsub_rn(phx, ch.x), __fsub_rn(plx, cl.x));
    dy = __fadd_rn(__fsub_rn(phy, ch.y), __fsub_rn(ply, cl.y));
    dz = __fadd_rn(__fsub_rn(phz, ch.z), __fsub_rn(plz, cl.z));
    return __fmaf_rn(dx, dx, __fmaf_rn(dy, dy, __fmul_rn(dz, dz)));
}

__device__ __forceinline__ void split2f(double x, float& hi, float& lo) {
    hi = __double2float_rn(x);
    lo = __double2float_rn(x - (double)hi);
}

// NP node pairs of one tier (layout in nb_internal.h: s = centroid - node, so the
// node-to-point vector is d + s) with the packed FP32x2 instructions: each instruction
// advances two nodes, lane x the first of a pair and lane y the second.
template <int NP>
__device__ __forceinline__ void node_pairs(const float4* __restrict__ nd, float2 dx, float2 dy, float2 dz,
                                           float2& ph, float2& ex, float2& ey, float2& ez) {
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        const float4 u = nd[2 * i], v = nd[2 * i + 1];
        const float2 rx = __fadd2_rn(dx, make_float2(u.x, u.y));
        const float2 ry = __fadd2_rn(dy, make_float2(u.z, u.w));
        const float2 rz = __fadd2_rn(dz, make_float2(v.x, v.y));
        const float2 r2 = __ffma2_rn(rx, rx, __ffma2_rn(ry, ry, __fmul2_rn(rz, rz)));
        const float2 ri = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
        const float2 wr = __fmul2_rn(make_float2(v.z, v.w), ri);
        const float2 wr3 = __fmul2_rn(wr, __fmul2_rn(ri, ri));
        ph = __fadd2_rn(ph, wr);
        ex = __ffma2_rn(wr3, rx, ex);
        ey = __ffma2_rn(wr3, ry, ey);
        ez = __ffma2_rn(wr3, rz, ez);
    }
}

// Tier 0 with its two node pairs held in registers (loaded once per element).
__device__ __forceinline__ void pairs0_reg(const float4 (&q)[2 * kPairs0], float2 dx, float2 dy, float2 dz,
                                           float2& ph, float2& ex, float2& ey, float2& ez) {
    node_pairs<kPairs0>(q, dx, dy, dz, ph, ex, ey, ez);
}

// Raw FP64 sums (phi, E; before the factor ke) of one point.
struct __align__(16) Sum4 {
    double phi, x, y, z;
};
// far sums plus the error scales B_phi, B_E (raw, before the factor ke)
struct __align__(16) Sum6 {
    double phi, x, y, z, bphi, bE;
};
// far sums of the FP32 pass with its four FP32 error scales (bound_slot)
struct __align__(16) SumB {
    Sum4 s;
    float4 b;
};
__device__ __forceinline__ void add_sum(Sum4& t, const Sum4& c) {
    t.phi += c.phi;
    t.x += c.x;
    t.y += c.y;
    t.z += c.z;
}
__device__ __forceinline__ void add_sum(Sum6& t, const Sum6& c) {
    t.phi += c.phi;
    t.x += c.x;
    t.y += c.y;
    t.z += c.z;
    t.bphi += c.bphi;
    t.bE += c.bE;
}
__device__ __forceinline__ void add_sum(SumB& t, const SumB& c) {
    add_sum(t.s, c.s);
    t.b.x += c.b.x;
    t.b.y += c.b.y;
    t.b.z += c.b.z;
    t.b.w += c.b.w;
}
// The total of one point's np pieces (leaves or chunks), added along the summation tree by
// one warp: lane l adds the leaves of chunk l, then every lane adds the chunks in order.
template <class T>
__device__ __forceinline__ T split_reduce(const T* __restrict__ part, int64_t np, int leaf) {
    constexpr int kPer = kChunkEl / kLeafEl, kWords = sizeof(T) / 4;
    const int lane = threadIdx.x & 31;
    const int64_t nch = leaf ? (np + kPer - 1) / kPer : np;
    T tot{};
    for (int64_t c0 = 0; c0 < nch; c0 += 32) {
        const int64_t c = c0 + lane;
        T own{};
        if (c < nch) {
            if (leaf) {
                for (int64_t l = c * kPer; l < c * kPer + kPer && l < np; ++l) add_sum(own, part[l]);
            } else {
                own = part[c];
            }
        }
        const int m = (int)(nch - c0 < 32 ? nch - c0 : 32);
        for (int k = 0; k < m; ++k) {
            T v;
#pragma unroll
            for (int w = 0; w < kWords; ++w)
                reinterpret_cast<int*>(&v)[w] = __shfl_sync(0xffffffffu, reinterpret_cast<const int*>(&own)[w], k);
            add_sum(tot, v);
        }
    }
    return tot;
}

// Per-thread error scales of the far pass, raw (before the factor ke): (B_phi, B_E, the
// sums of squares of the terms b_j of B_phi and B_E, each term scaled by kScaleSq first).
// Positive sums, FP32 is ample.  They live in a shared-memory slot (read and written once
// per element) rather than in registers across the element loop; bound_reset() before a
// point's first range.
// The squares are taken of b_j * 2^33 (2^33 ~ ke): a term of 1e-19 .. 1e19 volts then
// squares to a normal FP32 number.
constexpr float kScaleSq = 8589934592.0f;  // 2^33
__device__ __forceinline__ float4* bound_slot() {
    __shared__ float4 s_bnd[kEvalThreads];
    return &s_bnd[threadIdx.x];
}
__device__ __forceinline__ void bound_reset() { *bound_slot() = make_float4(0.f, 0.f, 0.f, 0.f); }
// Per-thread slots of the chunk and of the total of far_sum, in shared memory too.
__device__ __forceinline__ SumB* chunk_slot() {
    __shared__ SumB s_chunk[kEvalThreads];
    return &s_chunk[threadIdx.x];
}
__device__ __forceinline__ SumB* total_slot() {
    __shared__ SumB s_total[kEvalThreads];
    return &s_total[threadIdx.x];
}

// Raw FP64 sums of the far pairs of one point over the elements [e0, e1).  Called by every
// thread of the block (shared-memory tiles); the inactive threads' sums are unused.
__device__ __forceinline__ Sum4 far_range(const GeomView& g, float phx, float phy, float phz, float plx, float ply,
                                          float plz, int64_t e0, int64_t e1) {
    const FarNodes* __restrict__ far = g.far;
    const float4* __restrict__ cjk = g.cjk;
    const double* __restrict__ sigma = g.sigma;
    const int nimg = g.nimg;
    const int tile_el = g.tile_el;
    __shared__ float4 s_f[kTileMax][2 * kPairs0];
    __shared__ float4 s_a[kTileMax][2 * kPairsA];
    __shared__ int s_na[kTileMax];
    __shared__ float4 s_hdr[kTileMax];
    __shared__ float2 s_sig[kTileMax];  // sigma_j (1 + wcorr_j) as hi + lo
    __shared__ float4 s_c[kCjkMax][2];  // image centroids: hi, lo

    float4* bslot = bound_slot();
    double aphi = 0.0, aEx = 0.0, aEy = 0.0, aEz = 0.0;
    for (int64_t base = e0; base < e1; base += tile_el) {
        const int cnt = (int)min((int64_t)tile_el, e1 - base);
        __syncthreads();
        constexpr int kA = 2 * kPairsA, kF = 2 * kPairs0;
        for (int i = threadIdx.x; i < cnt * kA; i += blockDim.x) s_a[i / kA][i % kA] = far[base + i / kA].a[i % kA];
        for (int i = threadIdx.x; i < cnt * kF; i += blockDim.x) s_f[i / kF][i % kF] = far[base + i / kF].f[i % kF];
        for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
            s_hdr[i] = far[base + i].hdr;
            s_na[i] = far[base + i].n_a;
            const double sd = fma(sigma[base + i], (double)far[base + i].wcorr, sigma[base + i]);
            const float sh = __double2float_rn(sd);
            s_sig[i] = make_float2(sh, __double2float_rn(sd - (double)sh));
        }
        const float4* src = cjk + 2 * base * nimg;
        for (int i = threadIdx.x; i < 2 * cnt * nimg; i += blockDim.x) s_c[i >> 1][i & 1] = src[i];
        __syncthreads();
        float gphi = 0.f, gx = 0.f, gy = 0.f, gz = 0.f;
        for (int jj = 0; jj < cnt; ++jj) {
            const float4 hdr = s_hdr[jj];
            const bool rect = s_na[jj] == kPairsA;
            const FarNodes* fj = far + base + jj;
            float4 q[2 * kPairs0];
#pragma unroll
            for (int i = 0; i < 2 * kPairs0; ++i) q[i] = s_f[jj][i];
            float2 lphi = make_float2(0.f, 0.f), lx = lphi, ly = lphi, lz = lphi;
            // four images per round, so that one's distance test overlaps another's roots (1e6 points of the
            // 9,996-element cell x 25 copies: 610 ms, 592 so; two images 602, eight blocks of 64
            // registers per SM instead of six of 80 594 alone and 604 with it)
#pragma unroll 4
            for (int k = 0; k < nimg; ++k) {
                float dx, dy, dz;
                const float d2 = pair_d2(phx, phy, phz, plx, ply, plz, s_c[jj * nimg + k][0], s_c[jj * nimg + k][1],
                                         dx, dy, dz);
                const float2 DX = make_float2(dx, dx), DY = make_float2(dy, dy), DZ = make_float2(dz, dz);
                if (d2 >= hdr.x) {
                    pairs0_reg(q, DX, DY, DZ, lphi, lx, ly, lz);
                } else if (d2 >= hdr.y) {
                    if (rect)
                        node_pairs<kPairsA>(s_a[jj], DX, DY, DZ, lphi, lx, ly, lz);
                    else
                        node_pairs<3>(s_a[jj], DX, DY, DZ, lphi, lx, ly, lz);
                } else if (d2 >= hdr.z) {
                    node_pairs<kPairsB>(fj->b, DX, DY, DZ, lphi, lx, ly, lz);
                } else if (d2 >= hdr.w) {
                    node_pairs<kPairsC>(fj->c, DX, DY, DZ, lphi, lx, ly, lz);
                }
                // nearer pairs: k_eval_near
            }
            const float2 sg = s_sig[jj];
            const float s = sg.x;
            const float fphi = lphi.x + lphi.y, fx = lx.x + lx.y, fy = ly.x + ly.y, fz = lz.x + lz.y;
            // sigma in two floats: a density that is uniform over many elements (a plane far
            // from the structure) would otherwise carry one FP32 rounding error for all of them
            gphi = fmaf(s, fphi, fmaf(sg.y, fphi, gphi));
            gx = fmaf(s, fx, fmaf(sg.y, fx, gx));
            gy = fmaf(s, fy, fmaf(sg.y, fy, gy));
            gz = fmaf(s, fz, fmaf(sg.y, fz, gz));
            float4 b = *bslot;
            const float t0 = fabsf(s) * fabsf(fphi), t1 = fabsf(s) * (fabsf(fx) + fabsf(fy) + fabsf(fz));
            const float q0 = t0 * kScaleSq, q1 = t1 * kScaleSq;
            b.x += t0;
            b.y += t1;
            b.z = fmaf(q0, q0, b.z);
            b.w = fmaf(q1, q1, b.w);
            *bslot = b;
            if ((jj % kGroup) == kGroup - 1 || jj == cnt - 1) {
                aphi += (double)gphi;
                aEx += (double)gx;
                aEy += (double)gy;
                aEz += (double)gz;
                gphi = gx = gy = gz = 0.f;
            }
        }
    }
    return Sum4{aphi, aEx, aEy, aEz};
}

__device__ __forceinline__ void load_point_2f(const double* __restrict__ pts, int64_t p, bool active, float& phx,
                                              float& phy, float& phz, float& plx, float& ply, float& plz) {
    double Px = 0.0, Py = 0.0, Pz = 0.0;
    if (active) {
        Px = pts[3 * p];
        Py = pts[3 * p + 1];
        Pz = pts[3 * p + 2];
    }
    split2f(Px, phx, plx);
    split2f(Py, phy, ply);
    split2f(Pz, phz, plz);
}

// Stores ke * sum for point p.  A point with a non-finite coordinate has no field: it gets
// NaN in both precisions (the FP32 tiers would otherwise fail every distance test for it
// and leave zeros).  Its coordinates are read again here rather than kept in a register
// through the element loop.
template <class S>
__device__ __forceinline__ void store_far(const double* __restrict__ pts, double* __restrict__ phi,
                                          double* __restrict__ E, int64_t p, const S& s) {
    const double ke = 1.0 / (4.0 * kPi * kEps0);
    const bool finite = isfinite(pts[3 * p]) && isfinite(pts[3 * p + 1]) && isfinite(pts[3 * p + 2]);
    const double f = finite ? ke : __longlong_as_double(0x7ff8000000000000ll);
    if (phi) phi[p] = f * s.phi;
    if (E) {
        E[3 * p] = f * s.x;
        E[3 * p + 1] = f * s.y;
        E[3 * p + 2] = f * s.z;
    }
}

// ke * (B_phi, B_E, S_phi, S_E) of point p (the FP32 pass's error scales, V and V/m) from
// the raw sums of bound_slot()
__device__ __forceinline__ void store_bound(float4* __restrict__ bound, int64_t p, float4 b) {
    const double ke = 1.0 / (4.0 * kPi * kEps0);
    const double inv = 1.0 / (double)kScaleSq;
    if (bound)
        bound[p] = make_float4((float)(ke * b.x), (float)(ke * b.y), (float)(ke * inv * sqrt((double)b.z)),
                               (float)(ke * inv * sqrt((double)b.w)));
}

// The far sums and scales of one point over the elements [e0, e1) (whole pieces of the
// summation tree), left in total_slot(); every thread of the block takes part.
__device__ __forceinline__ void far_sum(const GeomView& g, float phx, float phy, float phz, float plx, float ply,
                                        float plz, int64_t e0, int64_t e1) {
    SumB* tot = total_slot();
    SumB* ch = chunk_slot();
    *tot = SumB{};
    for (int64_t c0 = e0; c0 < e1; c0 += kChunkEl) {
        const int64_t c1 = min(c0 + (int64_t)kChunkEl, e1);
        *ch = SumB{};
        for (int64_t l = c0; l < c1; l += kLeafEl) {
            bound_reset();
            SumB leaf;
            leaf.s = far_range(g, phx, phy, phz, plx, ply, plz, l, min(l + (int64_t)kLeafEl, c1));
            leaf.b = *bound_slot();
            add_sum(*ch, leaf);
        }
        add_sum(*tot, *ch);
    }
}

// Far part (FP32 tiers) of `count` targets over every element; writes ke * sum (overwrites
// phi / E).  Thread t takes point idx[base + t] (or base + t when idx is null) of pts / phi /
// E.  `bound` (may be null) receives ke * (B_phi, B_E, S_phi, S_E) per point.
__device__ __forceinline__ void far_block(const GeomView& g, const double* __restrict__ pts,
                                          const int32_t* __restrict__ idx, int64_t base, int count,
                                          double* __restrict__ phi, double* __restrict__ E,
                                          float4* __restrict__ bound) {
    const bool active = (int)threadIdx.x < count;
    const int64_t p = active ? (idx ? (int64_t)idx[base + threadIdx.x] : base + threadIdx.x) : 0;
    float phx, phy, phz, plx, ply, plz;
    load_point_2f(pts, p, active, phx, phy, phz, plx, ply, plz);
    far_sum(g, phx, phy, phz, plx, ply, plz, 0, g.n_el);
    if (active) {
        store_far(pts, phi, E, p, total_slot()->s);
        store_bound(bound, p, total_slot()->b);
    }
}

// The near pairs of the target (Px, Py, Pz) (ph, pl: its two floats), by one warp.  The image centroids in
// the 27 cells around the point are tested 32 at a time (a row of three cells is contiguous in
// cell_items), the near ones are queued in `queue` (kNearQueue entries of shared memory of the warp)
// and handed out 32 at a time: eval(live, jk) by every lane.  An FP64 instruction holds the SM's FP64 pipe
// as long for one lane as for 32, so a lane that met its near pairs one by one (a thread per point)
// made the pipe do mostly empty work and left one point's pairs in one serial chain (200,000
// points: 8.6 ms a thread per point, 1.4 ms a warp).  near2 gives the squared near radius of an
// element.  The order of the pairs depends on the point and the tables only.
constexpr int kNearQueue = 64;
template <class Near2, class Eval>
__device__ __forceinline__ void near_pairs_warp(double Px, double Py, double Pz, float phx, float phy, float phz,
                                                float plx, float ply, float plz, const float4* __restrict__ cjk,
                                                const NearGrid& grid, const int32_t* __restrict__ cell_start,
                                                const int32_t* __restrict__ cell_items, int nimg, const Near2& near2,
                                                int32_t* __restrict__ queue, const Eval& eval) {
    const int lane = threadIdx.x & 31;
    // cell of the point, clamped (a point more than one cell outside has no near pair)
    int cc[3];
    const double P[3] = {Px, Py, Pz};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double f = floor((P[a] - grid.origin[a]) * grid.inv_h);
        f = fmin(fmax(f, -2.0), (double)grid.dims[a] + 1.0);
        cc[a] = (int)f;
    }
    const int x0 = max(cc[0] - 1, 0), x1 = min(cc[0] + 1, grid.dims[0] - 1);
    int row = 0, nq = 0;  // rows (y, z) of the neighbourhood taken so far; queued pairs
    int32_t it = 0, end = 0;
    bool more = x0 <= x1;
    while (more || nq > 0) {
        while (more && nq < 32) {
            if (it >= end) {
                if (row == 9) {
                    more = false;
                    break;
                }
                const int y = cc[1] - 1 + row % 3, z = cc[2] - 1 + row / 3;
                ++row;
                if (y < 0 || y >= grid.dims[1] || z < 0 || z >= grid.dims[2]) continue;
                const int64_t cell = ((int64_t)z * grid.dims[1] + y) * grid.dims[0];
                it = cell_start[cell + x0];
                end = cell_start[cell + x1 + 1];
                continue;
            }
            bool hit = false;
            int32_t jk = 0;
            if (it + lane < end) {
                jk = cell_items[it + lane];
                float dx, dy, dz;
                const float d2 = pair_d2(phx, phy, phz, plx, ply, plz, cjk[2 * (int64_t)jk], cjk[2 * (int64_t)jk + 1],
                                         dx, dy, dz);
                hit = d2 < near2(jk / nimg);
            }
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            if (hit) queue[nq + __popc(m & ((1u << lane) - 1u))] = jk;
            nq += __popc(m);
            it += 32;
        }
        __syncwarp();
        const int take = min(nq, 32);
        if (take == 0) break;
        eval(lane < take, lane < take ? queue[lane] : 0);
        nq -= take;
        const int32_t rest = lane < nq ? queue[32 + lane] : 0;
        __syncwarp();
        if (lane < nq) queue[lane] = rest;
        __syncwarp();
    }
}

// Near part (FP64 closed forms) of target p, by one warp; adds ke * sum to phi[p] / E[p].
template <class Near2>
__device__ __forceinline__ void near_point_warp(const Elem* __restrict__ el, const double* __restrict__ sigma,
                                                const float4* __restrict__ cjk, const NearGrid& grid,
                                                const int32_t* __restrict__ cell_start,
                                                const int32_t* __restrict__ cell_items, const ImageTable& img,
                                                const Near2& near2, const double* __restrict__ pts, int64_t p,
                                                double* __restrict__ phi, double* __restrict__ E,
                                                int32_t* __restrict__ queue) {
    const int nimg = img.n;
    const double Px = pts[3 * p], Py = pts[3 * p + 1], Pz = pts[3 * p + 2];
    float phx, phy, phz, plx, ply, plz;
    split2f(Px, phx, plx);
    split2f(Py, phy, ply);
    split2f(Pz, phz, plz);
    double aphi = 0.0, aEx = 0.0, aEy = 0.0, aEz = 0.0;
    bool any = false;
    near_pairs_warp(Px, Py, Pz, phx, phy, phz, plx, ply, plz, cjk, grid, cell_start, cell_items, nimg, near2, queue,
                    [&](bool live, int32_t jk) {
                        any = true;
                        if (!live) return;
                        const int32_t j = jk / nimg, k = jk - j * nimg;
                        const Elem& e = el[j];
                        double f, ux, uy, uz;
                        elem_local_f64(e, Px - img.t[k][0], Py - img.t[k][1], Pz - img.t[k][2], false, f, ux, uy, uz);
                        const double s = sigma[j];
                        aphi = __fma_rn(s, f, aphi);
                        aEx = __fma_rn(s, __fma_rn(ux, e.ex[0], __fma_rn(uy, e.ey[0], __dmul_rn(uz, e.ez[0]))), aEx);
                        aEy = __fma_rn(s, __fma_rn(ux, e.ex[1], __fma_rn(uy, e.ey[1], __dmul_rn(uz, e.ez[1]))), aEy);
                        aEz = __fma_rn(s, __fma_rn(ux, e.ex[2], __fma_rn(uy, e.ey[2], __dmul_rn(uz, e.ez[2]))), aEz);
                    });
    if (!any) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        aphi += __shfl_xor_sync(0xffffffffu, aphi, o);
        aEx += __shfl_xor_sync(0xffffffffu, aEx, o);
        aEy += __shfl_xor_sync(0xffffffffu, aEy, o);
        aEz += __shfl_xor_sync(0xffffffffu, aEz, o);
    }
    if ((threadIdx.x & 31) != 0) return;
    const double ke = 1.0 / (4.0 * kPi * kEps0);
    if (phi) phi[p] = __fma_rn(ke, aphi, phi[p]);
    if (E) {
        E[3 * p] = __fma_rn(ke, aEx, E[3 * p]);
        E[3 * p + 1] = __fma_rn(ke, aEy, E[3 * p + 1]);
        E[3 * p + 2] = __fma_rn(ke, aEz, E[3 * p + 2]);
    }
}

// squared near radii of the fill and of refinement level 2
struct NearFill {
    const FillEl* fe;
    __device__ __forceinline__ float operator()(int32_t j) const { return fe[j].hdr.z; }
};
// squared near radii of the FP32 pass
struct NearFar {
    const FarNodes* far;
    __device__ __forceinline__ float operator()(int32_t j) const { return far[j].hdr.w; }
};
__device__ __forceinline__ void near_point(const GeomView& g, const ImageTable& img, const double* __restrict__ pts,
                                           int64_t p, double* __restrict__ phi, double* __restrict__ E) {
    __shared__ int32_t s_queue[kEvalThreads / 32][kNearQueue];
    near_point_warp(g.el, g.sigma, g.cjk, g.grid, g.cell_start, g.cell_items, img, NearFar{g.far}, pts, p, phi, E,
                    s_queue[threadIdx.x >> 5]);
}

// Raw FP64 sums (before the factor ke) of the closed forms of one point over the elements
// [e0, e1) and all images.  Called by every thread of the block (shared-memory tiles).
__device__ __forceinline__ Sum4 f64_range(const Elem* __restrict__ el, const double* __restrict__ sigma, int64_t e0,
                                          int64_t e1, const ImageTable& img, double Px, double Py, double Pz) {
    __shared__ Tile64 s_t;
    double aphi = 0.0, aEx = 0.0, aEy = 0.0, aEz = 0.0;
    for (int64_t base = e0; base < e1; base += kTile64) {
        const int cnt = (int)min((int64_t)kTile64, e1 - base);
        load_tile64(s_t, el, base, cnt, img);
        for (int jj = 0; jj < cnt; ++jj) {
            const Elem& e = s_t.el[jj];
            double X0, Y0, Z0;
            to_local(e, __dsub_rn(Px, e.o[0]), __dsub_rn(Py, e.o[1]), __dsub_rn(Pz, e.o[2]), X0, Y0, Z0);
            double lphi = 0.0, lx = 0.0, ly = 0.0, lz = 0.0;
            for (int k = 0; k < img.n; ++k) {
                const double* tau = s_t.tau[jj][k];
                double f, gx, gy, gz;
                elem_at_f64<true, true>(e, s_t.edge[jj], __dsub_rn(X0, tau[0]), __dsub_rn(Y0, tau[1]),
                                        __dsub_rn(Z0, tau[2]), f, gx, gy, gz);
                lphi = __dadd_rn(lphi, f);
                lx = __dadd_rn(lx, gx);
                ly = __dadd_rn(ly, gy);
                lz = __dadd_rn(lz, gz);
            }
            const double s = sigma[base + jj];
            aphi = __fma_rn(s, lphi, aphi);
            aEx = __fma_rn(s, __fma_rn(lx, e.ex[0], __fma_rn(ly, e.ey[0], __dmul_rn(lz, e.ez[0]))), aEx);
            aEy = __fma_rn(s, __fma_rn(lx, e.ex[1], __fma_rn(ly, e.ey[1], __dmul_rn(lz, e.ez[1]))), aEy);
            aEz = __fma_rn(s, __fma_rn(lx, e.ex[2], __fma_rn(ly, e.ey[2], __dmul_rn(lz, e.ez[2]))), aEz);
        }
    }
    return Sum4{aphi, aEx, aEy, aEz};
}

// The same over whole pieces of the summation tree, left in total_slot()->s.
__device__ __forceinline__ void f64_sum(const Elem* __restrict__ el, const double* __restrict__ sigma, int64_t e0,
                                        int64_t e1, const ImageTable& img, double Px, double Py, double Pz) {
    Sum4* tot = &total_slot()->s;
    Sum4* ch = &chunk_slot()->s;
    *tot = Sum4{};
    for (int64_t c0 = e0; c0 < e1; c0 += kChunkEl) {
        const int64_t c1 = min(c0 + (int64_t)kChunkEl, e1);
        *ch = Sum4{};
        for (int64_t l = c0; l < c1; l += kLeafEl)
            add_sum(*ch, f64_range(el, sigma, l, min(l + (int64_t)kLeafEl, c1), img, Px, Py, Pz));
        add_sum(*tot, *ch);
    }
}

// FP64 closed forms for every pair of `count` targets (overwrites phi / E).
__device__ __forceinline__ void f64_block(const Elem* __restrict__ el, const double* __restrict__ sigma, int64_t n_el,
                                          const ImageTable& img, const double* __restrict__ pts, int count,
                                          double* __restrict__ phi, double* __restrict__ E) {
    const int p = threadIdx.x;
    const bool active = p < count;
    double Px = 0.0, Py = 0.0, Pz = 0.0;
    if (active) {
        Px = pts[3 * p];
        Py = pts[3 * p + 1];
        Pz = pts[3 * p + 2];
    }
    f64_sum(el, sigma, 0, n_el, img, Px, Py, Pz);
    if (active) store_far(pts, phi, E, p, total_slot()->s);
}

}  // namespace nb
