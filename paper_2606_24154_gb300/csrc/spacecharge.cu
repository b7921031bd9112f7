// spacecharge.cu -- direct space-charge sums (Sec. 4.2, Alg. 2) and the carrier drift
// step of the dynamic update (Sec. 4.3, Alg. 4).
//
//   phi_t = ke sum_{c != self(t)} q_c / sqrt(r^2 + s^2)
//   E_t   = ke sum_{c != self(t)} q_c (x_t - x_c) / (r^2 + s^2)^{3/2}
//
// The paper launches one kernel per field point with a grid-stride loop over charges,
// a shared-memory tree and one atomicAdd per block.  Here all targets are evaluated in
// one launch as a tiled all-pairs sum: one thread per target, source tiles staged in
// shared memory, a fixed summation order (no atomics, bit-reproducible).
//
// Mixed precision: carriers are stored as two floats per coordinate (hi = fl(x),
// lo = fl(x - hi)).  x_t - x_c = (hi_t - hi_c) + (lo_t - lo_c): for nearby carriers
// hi_t - hi_c is exact (Sterbenz), so the difference keeps FP64 accuracy where it
// matters (near pairs) while every operation is FP32; the rest of the pair term is
// FP32 with rsqrt.  Runs of 32 sources are summed in FP32 and added to two-float
// (hi + lo) running totals with an error-free two-sum; each thread takes two targets in
// the lanes of the packed FP32x2 instructions.
#include <cooperative_groups.h>

#include <cfloat>

#include "influence.cuh"

namespace nb {

namespace {

constexpr int kSCThreads = 256;
constexpr int kFlush = 32;

struct __align__(16) Src64 {
    double x, y, z, w;  // position and charge
};

__global__ void __launch_bounds__(kSCThreads) k_sc_f64(const double* __restrict__ src, const double* __restrict__ q,
                                                       int64_t nsrc, const double* __restrict__ tgt, int64_t ntgt,
                                                       int exclude_self, double s2, double ke, int accumulate,
                                                       double* __restrict__ phi, double* __restrict__ E) {
    __shared__ Src64 ss[kSCThreads];
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool active = t < ntgt;
    double x = 0, y = 0, z = 0;
    if (active) {
        x = tgt[3 * t];
        y = tgt[3 * t + 1];
        z = tgt[3 * t + 2];
    }
    double ph = 0.0, ex = 0.0, ey = 0.0, ez = 0.0;
    for (int64_t base = 0; base < nsrc; base += kSCThreads) {
        __syncthreads();
        const int64_t c = base + threadIdx.x;
        if (c < nsrc) ss[threadIdx.x] = Src64{src[3 * c], src[3 * c + 1], src[3 * c + 2], q[c]};
        __syncthreads();
        const int cnt = (int)min((int64_t)kSCThreads, nsrc - base);
        for (int k = 0; k < cnt; ++k) {
            const Src64 s = ss[k];
            const double dx = x - s.x, dy = y - s.y, dz = z - s.z;
            const double r2 = fma(dx, dx, fma(dy, dy, fma(dz, dz, s2)));
            const double ri = 1.0 / sqrt(r2);
            double qq = s.w;
            if (exclude_self && base + k == t) qq = 0.0;
            const double qr = qq * ri;
            const double qr3 = qr * ri * ri;
            ph += qr;
            ex = fma(qr3, dx, ex);
            ey = fma(qr3, dy, ey);
            ez = fma(qr3, dz, ez);
        }
    }
    if (!active) return;
    if (accumulate) {
        if (phi) phi[t] += ke * ph;
        if (E) {
            E[3 * t] += ke * ex;
            E[3 * t + 1] += ke * ey;
            E[3 * t + 2] += ke * ez;
        }
    } else {
        if (phi) phi[t] = ke * ph;
        if (E) {
            E[3 * t] = ke * ex;
            E[3 * t + 1] = ke * ey;
            E[3 * t + 2] = ke * ez;
        }
    }
}

// Two-float split of carriers: hq = (hi.x, hi.y, hi.z, q), lo = (lo.x, lo.y, lo.z, 0).
__global__ void k_split2f(const double* __restrict__ pos, const double* __restrict__ q, int64_t n,
                          float4* __restrict__ hq, float4* __restrict__ lo) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x = pos[3 * i], y = pos[3 * i + 1], z = pos[3 * i + 2];
    const float hx = (float)x, hy = (float)y, hz = (float)z;
    hq[i] = make_float4(hx, hy, hz, (float)q[i]);
    lo[i] = make_float4((float)(x - hx), (float)(y - hy), (float)(z - hz), 0.f);
}

// Mixed sum: each thread takes P pairs of targets, a pair in the two lanes of the packed FP32x2
// instructions; a source tile is staged in shared memory with every value negated and
// duplicated into both lanes, so that a pair (target, source) costs the same rounded
// operations as the scalar form
//   d = (t_hi - s_hi) + (t_lo - s_lo),  r^2 = d.d + s^2,  q / r,  q d / r^3
// at half the issue slots (19 lane operations and one MUFU root).  Partial sums over kFlush sources
// are added to running totals kept as two floats (hi + lo, error-free two-sum), so no FP64
// instruction runs per source; the totals are converted to FP64 once per target.
//
// With SPLIT > 1 a cluster of SPLIT blocks shares a tile of targets: each sums a run of the sources, and
// the runs' totals are added in FP64 in the order of the runs through distributed shared memory,
// so the sums need neither scratch nor atomics.  The runs depend on the number of
// sources alone, and P does not enter the arithmetic: a target's bits do not depend on the others.
// Bound by the FP32 pipe with P = 2 (P = 1: by the four broadcast loads per source, 14 cycles of the
// shared-memory port against 9.5 of the FP32 pipe), given enough warps: 20,000 x 20,000 took 1.26 ms with
// one block per tile and P = 1, 0.40 ms in clusters of 8; 100,000 x 100,000 9.8 and 6.6 ms (4.8 ms
// at the FP32 pipe's rate); 100,000 sources at one target 6.3 and 0.46 ms.
constexpr int kSCT = 128;     // threads of a block
constexpr int kSCSrc = 256;   // sources of a staged tile
constexpr int kSCUnit = 128;  // the runs are whole units
constexpr int kSCSplit = 8;
constexpr int64_t kSCSplitFrom = 1024;

struct F2Acc {  // two-float running total per lane: value = hi + lo
    float2 hi, lo;
};

__device__ __forceinline__ void two_sum_add(float& hi, float& lo, float x) {
    const float s = __fadd_rn(hi, x);
    const float bb = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(x, bb));
    hi = s;
    lo = __fadd_rn(lo, e);
}

__device__ __forceinline__ void acc_add(F2Acc& a, float2 x) {
    two_sum_add(a.hi.x, a.lo.x, x.x);
    two_sum_add(a.hi.y, a.lo.y, x.y);
}

// NORMAL: r^2 >= s^2 >= FLT_MIN, so the root needs no scaling of subnormal arguments (about eight
// issue slots of 46 per pair of lanes; the same bits).
template <bool SELF, bool NORMAL, int P>
__device__ __forceinline__ void sc_run(const float4* __restrict__ A, const float4* __restrict__ B,
                                       const float4* __restrict__ C, const float2* __restrict__ D, int k0, int k1,
                                       const float2 (&th)[P][3], const float2 (&tl)[P][3], float2 s2,
                                       const int (&self)[2 * P], float2 (&ph)[P], float2 (&ex)[P], float2 (&ey)[P],
                                       float2 (&ez)[P]) {
#pragma unroll(4 / P)
    for (int k = k0; k < k1; ++k) {
        const float4 a = A[k], b = B[k], c = C[k];
        const float2 d = D[k];
#pragma unroll
        for (int h = 0; h < P; ++h) {
            const float2 dx =
                __fadd2_rn(__fadd2_rn(th[h][0], make_float2(a.x, a.y)), __fadd2_rn(tl[h][0], make_float2(c.x, c.y)));
            const float2 dy =
                __fadd2_rn(__fadd2_rn(th[h][1], make_float2(a.z, a.w)), __fadd2_rn(tl[h][1], make_float2(c.z, c.w)));
            const float2 dz = __fadd2_rn(__fadd2_rn(th[h][2], make_float2(b.x, b.y)), __fadd2_rn(tl[h][2], d));
            const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, s2)));
            const float2 ri = NORMAL ? make_float2(rsqrt_normal(r2.x), rsqrt_normal(r2.y))
                                     : make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
            float2 qq = make_float2(b.z, b.w);
            if (SELF) {
                if (k == self[2 * h]) qq.x = 0.f;
                if (k == self[2 * h + 1]) qq.y = 0.f;
            }
            const float2 qr = __fmul2_rn(qq, ri);
            const float2 qr3 = __fmul2_rn(qr, __fmul2_rn(ri, ri));
            ph[h] = __fadd2_rn(ph[h], qr);
            ex[h] = __ffma2_rn(qr3, dx, ex[h]);
            ey[h] = __ffma2_rn(qr3, dy, ey[h]);
            ez[h] = __ffma2_rn(qr3, dz, ez[h]);
        }
    }
}

__device__ __forceinline__ void load_target_2f(const double* __restrict__ tgt, int64_t t, bool active, float& hx,
                                               float& hy, float& hz, float& lx, float& ly, float& lz) {
    double x = 0, y = 0, z = 0;
    if (active) {
        x = tgt[3 * t];
        y = tgt[3 * t + 1];
        z = tgt[3 * t + 2];
    }
    hx = (float)x;
    hy = (float)y;
    hz = (float)z;
    lx = (float)(x - hx);
    ly = (float)(y - hy);
    lz = (float)(z - hz);
}

__device__ __forceinline__ void store_target(int64_t t, int accumulate, double ke, double ph, double ex, double ey,
                                             double ez, double* __restrict__ phi, double* __restrict__ E) {
    if (accumulate) {
        if (phi) phi[t] += ke * ph;
        if (E) {
            E[3 * t] += ke * ex;
            E[3 * t + 1] += ke * ey;
            E[3 * t + 2] += ke * ez;
        }
    } else {
        if (phi) phi[t] = ke * ph;
        if (E) {
            E[3 * t] = ke * ex;
            E[3 * t + 1] = ke * ey;
            E[3 * t + 2] = ke * ez;
        }
    }
}

// Targets given as FP64 (split in-kernel); sources as two-float (hi, lo) arrays.  Grid: SPLIT blocks
// per tile of 2 P kSCT targets, which are clusters for SPLIT > 1.
template <int P, int SPLIT>
__device__ __forceinline__ void sc_mixed(const float4* __restrict__ shq, const float4* __restrict__ slo, int64_t nsrc,
                                         const double* __restrict__ tgt, int64_t ntgt, int exclude_self, float s2,
                                         double ke, int accumulate, double* __restrict__ phi, double* __restrict__ E) {
    constexpr int kTile = 2 * P * kSCT;
    struct Stage {
        float4 A[kSCSrc], B[kSCSrc], C[kSCSrc];
        float2 D[kSCSrc];
    };
    __shared__ union {
        Stage st;
        double part[SPLIT > 1 ? 4 * kTile : 1];
    } sm;
    const int run = SPLIT > 1 ? (int)(blockIdx.x % SPLIT) : 0;
    const int64_t first = (int64_t)(blockIdx.x / SPLIT) * kTile;
    float2 th[P][3], tl[P][3];
#pragma unroll
    for (int h = 0; h < P; ++h) {
        float hx[2], hy[2], hz[2], lx[2], ly[2], lz[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int64_t t = first + threadIdx.x + (2 * h + q) * kSCT;
            load_target_2f(tgt, t, t < ntgt, hx[q], hy[q], hz[q], lx[q], ly[q], lz[q]);
        }
        th[h][0] = make_float2(hx[0], hx[1]), th[h][1] = make_float2(hy[0], hy[1]), th[h][2] = make_float2(hz[0], hz[1]);
        tl[h][0] = make_float2(lx[0], lx[1]), tl[h][1] = make_float2(ly[0], ly[1]), tl[h][2] = make_float2(lz[0], lz[1]);
    }
    const float2 s22 = make_float2(s2, s2);
    const bool normal = s2 >= FLT_MIN;
    const float2 zero = make_float2(0.f, 0.f);
    F2Acc aph[P], aex[P], aey[P], aez[P];
#pragma unroll
    for (int h = 0; h < P; ++h) aph[h] = aex[h] = aey[h] = aez[h] = F2Acc{zero, zero};
    const int64_t units = (nsrc + kSCUnit - 1) / kSCUnit;
    const int64_t c0 = SPLIT > 1 ? units * run / SPLIT * kSCUnit : 0;
    const int64_t c1 = SPLIT > 1 ? min(nsrc, units * (run + 1) / SPLIT * kSCUnit) : nsrc;
    for (int64_t base = c0; base < c1; base += kSCSrc) {
        const int cnt = (int)min((int64_t)kSCSrc, c1 - base);
        __syncthreads();
        for (int i = threadIdx.x; i < cnt; i += kSCT) {
            const float4 h = shq[base + i], l = slo[base + i];
            sm.st.A[i] = make_float4(-h.x, -h.x, -h.y, -h.y);
            sm.st.B[i] = make_float4(-h.z, -h.z, h.w, h.w);
            sm.st.C[i] = make_float4(-l.x, -l.x, -l.y, -l.y);
            sm.st.D[i] = make_float2(-l.z, -l.z);
        }
        __syncthreads();
        // the block's own carriers (targets are the sources in order): source `self` of this tile
        const bool own = exclude_self && base < first + kTile && first < base + cnt;
        int self[2 * P];
#pragma unroll
        for (int q = 0; q < 2 * P; ++q) self[q] = own ? (int)(first - base) + (int)threadIdx.x + q * kSCT : -1;
        // FP32 partial sums over kFlush sources: the +/- charges cancel, so longer FP32
        // runs would lose the result in the partial sums' rounding
        for (int sub = 0; sub < cnt; sub += kFlush) {
            const int m = min(kFlush, cnt - sub);
            float2 fph[P], fex[P], fey[P], fez[P];
#pragma unroll
            for (int h = 0; h < P; ++h) fph[h] = fex[h] = fey[h] = fez[h] = zero;
            bool hit = false;
#pragma unroll
            for (int q = 0; q < 2 * P; ++q) hit |= self[q] >= sub && self[q] < sub + m;
            if (hit)
                sc_run<true, false, P>(sm.st.A, sm.st.B, sm.st.C, sm.st.D, sub, sub + m, th, tl, s22, self, fph, fex, fey, fez);
            else if (normal)
                sc_run<false, true, P>(sm.st.A, sm.st.B, sm.st.C, sm.st.D, sub, sub + m, th, tl, s22, self, fph, fex,
                                       fey, fez);
            else
                sc_run<false, false, P>(sm.st.A, sm.st.B, sm.st.C, sm.st.D, sub, sub + m, th, tl, s22, self, fph, fex,
                                        fey, fez);
#pragma unroll
            for (int h = 0; h < P; ++h) {
                acc_add(aph[h], fph[h]);
                acc_add(aex[h], fex[h]);
                acc_add(aey[h], fey[h]);
                acc_add(aez[h], fez[h]);
            }
        }
    }
    auto total = [](const F2Acc& a, int q) {
        return q ? (double)a.hi.y + (double)a.lo.y : (double)a.hi.x + (double)a.lo.x;
    };
    if constexpr (SPLIT == 1) {
#pragma unroll
        for (int q = 0; q < 2 * P; ++q) {
            const int64_t t = first + threadIdx.x + q * kSCT;
            if (t < ntgt)
                store_target(t, accumulate, ke, total(aph[q / 2], q & 1), total(aex[q / 2], q & 1),
                             total(aey[q / 2], q & 1), total(aez[q / 2], q & 1), phi, E);
        }
    } else {
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 2 * P; ++q) {
            double* o = sm.part + 4 * (threadIdx.x + q * kSCT);
            o[0] = total(aph[q / 2], q & 1), o[1] = total(aex[q / 2], q & 1);
            o[2] = total(aey[q / 2], q & 1), o[3] = total(aez[q / 2], q & 1);
        }
        cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
        cl.sync();
        // the tile's targets dealt to the blocks
        for (int i = run * (kTile / SPLIT) + threadIdx.x; i < (run + 1) * (kTile / SPLIT); i += kSCT) {
            double v[4] = {0.0, 0.0, 0.0, 0.0};
            for (int r = 0; r < SPLIT; ++r) {
                const double2* o = reinterpret_cast<const double2*>(cl.map_shared_rank(sm.part, r)) + 2 * i;
                const double2 a = o[0], b = o[1];
                v[0] += a.x, v[1] += a.y, v[2] += b.x, v[3] += b.y;
            }
            if (first + i < ntgt) store_target(first + i, accumulate, ke, v[0], v[1], v[2], v[3], phi, E);
        }
        cl.sync();  // the other blocks read this block's shared memory
    }
}

template <int P>
__global__ void __launch_bounds__(kSCT, 4) k_sc_mixed(const float4* __restrict__ shq, const float4* __restrict__ slo,
                                                      int64_t nsrc, const double* __restrict__ tgt, int64_t ntgt,
                                                      int exclude_self, float s2, double ke, int accumulate,
                                                      double* __restrict__ phi, double* __restrict__ E) {
    sc_mixed<P, 1>(shq, slo, nsrc, tgt, ntgt, exclude_self, s2, ke, accumulate, phi, E);
}
template <int P>
__global__ void __cluster_dims__(kSCSplit, 1, 1) __launch_bounds__(kSCT, 4)
    k_sc_mixed_split(const float4* __restrict__ shq, const float4* __restrict__ slo, int64_t nsrc,
                     const double* __restrict__ tgt, int64_t ntgt, int exclude_self, float s2, double ke,
                     int accumulate, double* __restrict__ phi, double* __restrict__ E) {
    sc_mixed<P, kSCSplit>(shq, slo, nsrc, tgt, ntgt, exclude_self, s2, ke, accumulate, phi, E);
}

// b_i -= phi_sc(c_i) on conductor rows, b_i -= n_i . E_sc(c_i) on interface rows.
__global__ void k_rhs_sc(const Elem* __restrict__ el, int64_t n, const double* __restrict__ phi,
                         const double* __restrict__ E, double* __restrict__ b) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Elem& e = el[i];
    if (e.bc == NEBEM_CONDUCTOR)
        b[i] -= phi[i];
    else
        b[i] -= e.ey[0] * E[3 * i] + e.ey[1] * E[3 * i + 1] + e.ey[2] * E[3 * i + 2];
}

__global__ void k_centroids(const Elem* __restrict__ el, int64_t n, double* __restrict__ c) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    c[3 * i] = el[i].c[0];
    c[3 * i + 1] = el[i].c[1];
    c[3 * i + 2] = el[i].c[2];
}

// x_c += sign(q_c) mu E_c dt
__global__ void k_drift(double* __restrict__ pos, const double* __restrict__ q, const double* __restrict__ E,
                        int64_t n, double mu_dt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double s = (q[i] > 0.0) ? 1.0 : ((q[i] < 0.0) ? -1.0 : 0.0);
    const double f = s * mu_dt;
    pos[3 * i] += f * E[3 * i];
    pos[3 * i + 1] += f * E[3 * i + 1];
    pos[3 * i + 2] += f * E[3 * i + 2];
}

}  // namespace

cudaError_t launch_sc_split(const double* pos, const double* q, int64_t n, float4* hq, float4* lo, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_split2f<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pos, q, n, hq, lo);
    return cudaGetLastError();
}

cudaError_t launch_sc_eval(int precision, const double* src, const double* q, const float4* hq, const float4* lo,
                           int64_t nsrc, const double* tgt, int64_t ntgt, int exclude_self, double soft,
                           int accumulate, double* phi, double* E, cudaStream_t s) {
    if (ntgt == 0) return cudaSuccess;
    const double ke = 1.0 / (4.0 * kPi * kEps0);
    const unsigned blocks = (unsigned)((ntgt + kSCThreads - 1) / kSCThreads);
    if (precision == NEBEM_FP64)
        k_sc_f64<<<blocks, kSCThreads, 0, s>>>(src, q, nsrc, tgt, ntgt, exclude_self, soft * soft, ke, accumulate, phi,
                                               E);
    else {
        // Sources shared among the blocks of a cluster from kSCSplitFrom on: with 1,100 sources a call takes 13
        // us against 43 (1,100 targets), 39 against 44 (20,000) and 205 against 178 (200,000, where the blocks'
        // targets and totals cost more than the idle SMs; 275 against 315 with 2,000 sources).  Two pairs
        // of targets per thread where that leaves a block for every SM.
        int sms = 0;
        const cudaError_t e = sm_count(&sms);
        if (e != cudaSuccess) return e;
        const bool split = nsrc >= kSCSplitFrom;
        const int ns = split ? kSCSplit : 1;
        const bool wide = ntgt * ns >= (int64_t)sms * 2 * kSCT;
        const int64_t tile = (wide ? 4 : 2) * kSCT;
        const unsigned grid = (unsigned)((ntgt + tile - 1) / tile * ns);
        auto* k = split ? (wide ? k_sc_mixed_split<2> : k_sc_mixed_split<1>) : (wide ? k_sc_mixed<2> : k_sc_mixed<1>);
        k<<<grid, kSCT, 0, s>>>(hq, lo, nsrc, tgt, ntgt, exclude_self, (float)(soft * soft), ke, accumulate, phi, E);
    }
    return cudaGetLastError();
}

cudaError_t launch_rhs_sc(const Elem* el, int64_t n, const double* phi, const double* E, double* b, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_rhs_sc<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(el, n, phi, E, b);
    return cudaGetLastError();
}

cudaError_t launch_centroids(const Elem* el, int64_t n, double* c, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_centroids<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(el, n, c);
    return cudaGetLastError();
}

cudaError_t launch_drift(double* pos, const double* q, const double* E, int64_t n, double mu_dt, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_drift<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(pos, q, E, n, mu_dt);
    return cudaGetLastError();
}

}  // namespace nb
