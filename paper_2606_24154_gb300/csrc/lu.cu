// lu.cu -- dense LU with partial pivoting, triangular solves, residual and refinement
// helpers (Sec. 4.1, Alg. 1: the paper inverts K with an LU factorisation; here the
// factors are kept and applied by forward/back substitution instead of forming K^-1).
//
// Right-looking blocked LU, column-major, lda = n, panel width nb:
//   for each panel [k0, k0+nb):
//     per column j: pivot search (max |a|, lowest row index on ties) -> row swap
//                   inside the panel -> scale the column -> rank-1 update of the panel;
//     apply the panel's swaps to the other columns;
//     U12 = L11^-1 A12  (explicit inverse of the unit-lower nb x nb block, then a GEMM);
//     A22 -= L21 U12    (GEMM).
// A22 -= L21 U12 runs on the tensor cores in both precisions (lu_tc.cu, lu_tc64.cu).
// Templated on the element type: double (FP64 solves) and float (mixed solves, the
// FP64 iterative refinement lives in the caller).
#include <cooperative_groups.h>
#include <algorithm>
#include <climits>
#include <vector>

#include "nb_internal.h"

namespace nb {

namespace {

constexpr int kPivBlocks = 256;
constexpr int kPivThreads = 256;

// One launch per panel column j, fusing what would otherwise be three launches:
//   (a) for j > k0: scale column j-1 below its diagonal and apply its rank-1 update to
//       the panel columns (j-1, k1), each thread for its own rows i >= j;
//   (b) the partial pivot search of column j over the same rows (so a thread reads only
//       values it has just updated itself);
//   (c) the last block to finish (an atomic ticket, no waiting) reduces the partial maxima,
//       records the pivot and swaps rows j and p inside the panel columns.
// With do_pivot = 0 only (a) runs (the launch after the panel's last column).  The
// per-element arithmetic is that of the three separate steps, in the same order.
template <typename T>
__global__ void __launch_bounds__(kPivThreads, 2) k_panel_col(T* __restrict__ A, int64_t n, int64_t j, int64_t k0,
                                                            int64_t k1, int do_pivot, double* __restrict__ pval,
                                                            int64_t* __restrict__ pidx, int* __restrict__ ticket,
                                                            int32_t* __restrict__ piv, int* __restrict__ info) {
    __shared__ T urow[64];
    __shared__ double sv[kPivThreads];
    __shared__ int64_t si[kPivThreads];
    __shared__ bool last;
    const bool update = j > k0;
    const int64_t jm = j - 1;
    const int w = update ? (int)(k1 - j) : 0;  // columns (j-1, k1)
    T inv = (T)0;
    bool ok = true;
    if (update) {
        for (int c = threadIdx.x; c < w; c += blockDim.x) urow[c] = A[jm + (j + c) * n];
        const T d = A[jm + jm * n];
        ok = d != (T)0;
        inv = ok ? (T)1 / d : (T)0;
    }
    __syncthreads();
    double best = -1.0;
    int64_t bidx = INT64_MAX;
    for (int64_t i = j + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        T aj;  // A[i, j] after the update
        if (update && ok) {
            const T l = A[i + jm * n] * inv;
            A[i + jm * n] = l;
            // the row's panel values in batches of 16 independent loads (one memory round
            // trip per batch instead of one per column), then the updates
            T* row = A + i + j * n;
            aj = (T)0;
            for (int c0 = 0; c0 < w; c0 += 16) {
                T v[16];
#pragma unroll
                for (int q = 0; q < 16; ++q)
                    if (c0 + q < w) v[q] = row[(int64_t)(c0 + q) * n];
#pragma unroll
                for (int q = 0; q < 16; ++q)
                    if (c0 + q < w) {
                        v[q] -= l * urow[c0 + q];
                        row[(int64_t)(c0 + q) * n] = v[q];
                    }
                if (c0 == 0) aj = v[0];
            }
        } else {
            aj = A[i + j * n];
        }
        if (do_pivot) {
            const double v = fabs((double)aj);
            if (v > best || (v == best && i < bidx)) {
                best = v;
                bidx = i;
            }
        }
    }
    if (!do_pivot) return;
    sv[threadIdx.x] = best;
    si[threadIdx.x] = bidx;
    __syncthreads();
    for (int st = blockDim.x / 2; st > 0; st >>= 1) {
        if (threadIdx.x < st) {
            const double v = sv[threadIdx.x + st];
            const int64_t ix = si[threadIdx.x + st];
            if (v > sv[threadIdx.x] || (v == sv[threadIdx.x] && ix < si[threadIdx.x])) {
                sv[threadIdx.x] = v;
                si[threadIdx.x] = ix;
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        pval[blockIdx.x] = sv[0];
        pidx[blockIdx.x] = si[0];
        __threadfence();
        last = atomicAdd(ticket, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // final reduction over the blocks' partial maxima (lowest row index on ties)
    best = -1.0;
    bidx = INT64_MAX;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) {
        const double v = __ldcg(pval + b);
        const int64_t ix = __ldcg(pidx + b);
        if (v > best || (v == best && ix < bidx)) {
            best = v;
            bidx = ix;
        }
    }
    sv[threadIdx.x] = best;
    si[threadIdx.x] = bidx;
    __syncthreads();
    for (int st = blockDim.x / 2; st > 0; st >>= 1) {
        if (threadIdx.x < st) {
            const double v = sv[threadIdx.x + st];
            const int64_t ix = si[threadIdx.x + st];
            if (v > sv[threadIdx.x] || (v == sv[threadIdx.x] && ix < si[threadIdx.x])) {
                sv[threadIdx.x] = v;
                si[threadIdx.x] = ix;
            }
        }
        __syncthreads();
    }
    const int64_t p = (si[0] >= j && si[0] < n) ? si[0] : j;
    if (threadIdx.x == 0) {
        piv[j] = (int32_t)p;
        if (!(sv[0] > 0.0) && *info == 0) *info = (int)(j + 1);
        *ticket = 0;
    }
    if (p != j) {
        for (int64_t c = k0 + threadIdx.x; c < k1; c += blockDim.x) {
            const T a = __ldcg(A + j + c * n);
            A[j + c * n] = __ldcg(A + p + c * n);
            A[p + c * n] = a;
        }
    }
}

// The whole panel in one cooperative launch (all CTAs resident), FP32 and FP64.  CTA b holds rows
// [k0 + b R, k0 + (b+1) R) of the panel columns in shared memory (column-major, R rows); per
// column j of the panel:
//   (a) the rank-1 update of column j-1 on the rows below it (the per-element arithmetic of
//       k_panel_col), the columns dealt to groups of threads where the rows do not fill the block.
//       L's columns stay unscaled in shared memory, scaled where they are used and when they
//       are written back;
//   (b) each CTA finds its largest |a_ij| (lowest row on ties) and warp 0 publishes it: the row and
//       a 16-byte slot (magnitude, row index) of parity j & 1; the CTA that holds row j publishes
//       row j too.  Then the grid barrier: one acquire-release add to an arrival counter that
//       counts all arrivals of the factorisation, and polls of it until this column's total;
//   (c) thread q of every CTA reads slot q; the CTA reduces them to the pivot p, reads the pivot
//       row, and the holders of rows j and p swap them in shared memory.
// The slots alternate between two parities: a CTA writes slot j+1 only after it has passed
// barrier j, by which time every CTA has finished reading slot j-1.  A poll gives up after `limit`
// reads; the CTA records *err and leaves the panel (the host reports a timeout), and the others
// follow.
//
// Bound by latency: per column four block barriers and three L2 round trips in turn (arrival,
// slots, pivot row).  A column takes 2.7 us in FP32 (n = 9996; 3.4 with shuffles for the
// reductions, a barrier after each, L scaled and stored at once) and 3.1 us in FP64 (n = 6145;
// 5.1 with one thread per row and the reciprocal taken by every thread).  Polling the CTAs' tagged
// slots in place of the counter was slower on many CTAs (152: 3.9 us).
constexpr int kCoopThreads = 256;
constexpr int kCoopMaxG = kCoopThreads;  // one reading thread per CTA of the grid
constexpr long long kCoopSpinLimit = 1ll << 22;
// The kernels' shared-memory limits are set to one value each, whatever the call's size: a limit belongs to the
// function, and another thread's call of another size may be between its setting and its launches.
constexpr int kCoopSmemMax = 200 * 1024;

// A magnitude as it is compared: its bits (non-negative numbers order as their bits, and integer
// compares leave the FP64 pipe alone).  NaN never wins: -1.
template <typename T>
struct Mag;
template <>
struct Mag<float> {
    static __device__ __forceinline__ long long of(float a) {
        const int m = __float_as_int(a) & 0x7fffffff;
        return m <= 0x7f800000 ? m : -1;
    }
};
template <>
struct Mag<double> {
    static __device__ __forceinline__ long long of(double a) {
        const long long m = __double_as_longlong(a) & 0x7fffffffffffffffll;
        return m <= 0x7ff0000000000000ll ? m : -1;
    }
};

// rows a CTA holds at least: FP64 updates are bound by the FP64 pipe (one warp of rows), FP32 ones are not
template <typename T>
constexpr int64_t kCoopMinRows = sizeof(T) == 8 ? 32 : 64;

struct __align__(16) CoopSlot {
    long long key;
    int idx, pad;
};
template <typename T>
struct CoopScratch {
    CoopSlot slot[2][kCoopMaxG];
    alignas(16) T cand[2][kCoopMaxG][64];
    alignas(16) T srow[2][64];
    unsigned int bar;  // arrivals of the factorisation
    int err;
};

__device__ __forceinline__ int ld_acquire_i(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned int ld_acquire_u(const unsigned int* p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// largest key of the warp with the lowest index on ties, in every lane
__device__ __forceinline__ void warp_best(long long& key, int& idx) {
    const int hi = (int)(key >> 32);
    const int mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned int lo = hi == mh ? (unsigned int)key : 0u;
    const unsigned int ml = __reduce_max_sync(0xffffffffu, lo);
    const bool mine = hi == mh && (unsigned int)key == ml;
    idx = __reduce_min_sync(0xffffffffu, mine ? idx : INT_MAX);
    key = ((long long)mh << 32) | ml;
}

// CL: the grid is one cluster of kPanelCluster CTAs.  The slots are pushed into every CTA's shared memory, the
// rows are read from their holders' (distributed shared memory), and the cluster barrier, which needs no
// bound, takes the place of the counter: 2.2 us a column in FP64 (up to 1,536 rows), 1.7 to 2.1 in FP32 (up to 4,096).
constexpr int kPanelCluster = 16;

template <typename T, bool CL>
__device__ __forceinline__ void panel(T* __restrict__ A, int64_t n, int64_t k0, int64_t k1, int R,
                                      int32_t* __restrict__ piv, int* __restrict__ info, int* __restrict__ tmo,
                                      CoopScratch<T>* cs, unsigned int bar_base, long long limit) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (ld_acquire_i(&cs->err)) return;  // an earlier panel gave up: leave the matrix as it is
    const int w = (int)(k1 - k0);
    T* S = reinterpret_cast<T*>(smem_raw);  // R x w, column-major
    constexpr int kWarps = kCoopThreads / 32;
    __shared__ T prow[64], sinv[64];
    __shared__ long long wk[2][kWarps];
    __shared__ int wi[2][kWarps];
    __shared__ int s_fail;
    __shared__ CoopSlot c_slot[2][CL ? kPanelCluster : 1];  // CL: every CTA's slots, own candidate, own row j
    __shared__ T c_cand[2][CL ? 64 : 1], c_srow[2][CL ? 64 : 1];
    const int G = gridDim.x, b = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    const int64_t rb0 = k0 + (int64_t)b * R;
    const int nr = (int)max((int64_t)0, min((int64_t)R, n - rb0));
    if (tid == 0) s_fail = 0;
    for (int idx = tid; idx < nr * w; idx += kCoopThreads) {
        const int r = idx % nr, c = idx / nr;
        S[c * R + r] = A[(rb0 + r) + (k0 + c) * n];
    }
    // CL: the first column's slots go to the other CTAs' shared memory, which may be touched only once those
    // CTAs run (one that holds no rows gets here at once)
    if constexpr (CL)
        cg::this_cluster().sync();
    else
        __syncthreads();
    // thread -> row and group of columns: `step` rows at a time, `groups` column groups
    const int step = R <= kCoopThreads / 2 ? (R + 31) & ~31 : kCoopThreads;
    const int groups = kCoopThreads / step, grp = tid / step, row0 = tid - grp * step;
    // (key, index) of the block, in every thread, through buffer q
    auto block_best = [&](int q, long long& key, int& idx) {
        warp_best(key, idx);
        if (lane == 0) {
            wk[q][tid >> 5] = key;
            wi[q][tid >> 5] = idx;
        }
        __syncthreads();
        key = lane < kWarps ? wk[q][lane] : -1;
        idx = lane < kWarps ? wi[q][lane] : INT_MAX;
        warp_best(key, idx);
    };
    bool ok_piv = true;  // the previous pivot was nonzero
    for (int jj = 0; jj < w; ++jj) {
        const int64_t j = k0 + jj;
        const int par = jj & 1;
        // (a) column jj-1's rank-1 update, then this thread's candidate for column jj
        long long best = -1;
        int bidx = INT_MAX;
        const T inv = jj > 0 ? sinv[jj - 1] : (T)0;
        if (grp < groups)
            for (int r = row0; r < nr; r += step) {
                if (rb0 + r < j) continue;
                if (jj > 0 && ok_piv) {
                    const T l = S[(jj - 1) * R + r] * inv;
#pragma unroll 4
                    for (int c = jj + grp; c < w; c += groups) S[c * R + r] -= l * prow[c];
                }
                if (grp == 0) {
                    const long long v = Mag<T>::of(S[jj * R + r]);
                    if (v > best) {  // rows in increasing order: the first of equal ones stays
                        best = v;
                        bidx = (int)(rb0 + r);
                    }
                }
            }
        block_best(0, best, bidx);
        // (b) warp 0 publishes the candidate row (and row j), then the slot
        if (tid < 32) {
            const int mine = bidx != INT_MAX ? (int)(bidx - rb0) : -1;
            const bool own = j >= rb0 && j < rb0 + nr;
            T* cand = CL ? c_cand[par] : cs->cand[par][b];
            T* srow = CL ? c_srow[par] : cs->srow[par];
            for (int c = lane; c < w; c += 32) {
                cand[c] = mine >= 0 ? S[c * R + mine] : (T)0;
                if (own) srow[c] = S[c * R + (int)(j - rb0)];
            }
            if constexpr (CL) {
                if (lane < G)
                    *cg::this_cluster().map_shared_rank(&c_slot[par][b], lane) = CoopSlot{best, bidx, 0};
            }
            __syncwarp();
            if (!CL && lane == 0) {
                __stcg(reinterpret_cast<int4*>(&cs->slot[par][b]),
                       make_int4((int)best, (int)(best >> 32), bidx, 0));
                // the barrier: the release half publishes the warp's stores (cumulative over the
                // warp barrier), the acquire of the final count everyone's
                const unsigned int target = bar_base + (unsigned)(jj + 1) * (unsigned)G;
                unsigned int v;
                asm volatile("atom.add.acq_rel.gpu.u32 %0, [%1], 1;" : "=r"(v) : "l"(&cs->bar) : "memory");
                long long spins = 0;
                while (v + 1u < target && ld_acquire_u(&cs->bar) < target) {
                    // give up after the poll limit, or when another CTA has given up
                    if (++spins > limit || ((spins & 1023) == 0 && ld_acquire_i(&cs->err))) {
                        s_fail = 1;
                        break;
                    }
                    __nanosleep(20);
                }
            }
        }
        if constexpr (CL)
            cg::this_cluster().sync();
        else
            __syncthreads();
        // (c) every CTA's candidate
        best = -1;
        bidx = INT_MAX;
        if (CL && tid < G) {
            best = c_slot[par][tid].key;
            bidx = c_slot[par][tid].idx;
        } else if (!CL && tid < G) {
            const int4 q = __ldcg(reinterpret_cast<const int4*>(&cs->slot[par][tid]));
            best = ((long long)q.y << 32) | (unsigned int)q.x;
            bidx = q.z;
        }
        block_best(1, best, bidx);
        if (!CL && s_fail) {
            if (tid == 0) {
                atomicExch(&cs->err, 1);
                atomicExch(tmo, 1);
            }
            return;
        }
        // no candidate (a column of NaN): row j stays where it is
        const bool any = (int64_t)bidx >= j && (int64_t)bidx < n;
        const int64_t p = any ? (int64_t)bidx : j;
        if (tid < w) {
            auto row_j = [&]() {
                if constexpr (CL) return *cg::this_cluster().map_shared_rank(&c_srow[par][tid], (int)((j - k0) / R));
                return __ldcg(&cs->srow[par][tid]);
            };
            auto row_p = [&]() {
                if constexpr (CL) return *cg::this_cluster().map_shared_rank(&c_cand[par][tid], (int)((p - k0) / R));
                return __ldcg(&cs->cand[par][(int)((p - k0) / R)][tid]);
            };
            const T v = any ? row_p() : row_j();
            prow[tid] = v;
            if (j >= rb0 && j < rb0 + nr) S[tid * R + (int)(j - rb0)] = v;
            if (p != j && p >= rb0 && p < rb0 + nr) S[tid * R + (int)(p - rb0)] = row_j();
            // a zero pivot leaves its column unscaled and skips its update, as in k_panel_col
            if (tid == jj) sinv[jj] = v != (T)0 ? (T)1 / v : (T)1;
        }
        if (b == 0 && tid == 0) {
            piv[j] = (int32_t)p;
            if (!(best > 0) && *info == 0) *info = (int)(j + 1);
        }
        __syncthreads();
        ok_piv = prow[jj] != (T)0;
    }
    for (int idx = tid; idx < nr * w; idx += kCoopThreads) {
        const int r = idx % nr, c = idx / nr;
        const T v = S[c * R + r];
        A[(rb0 + r) + (k0 + c) * n] = rb0 + r > k0 + c ? v * sinv[c] : v;
    }
    if constexpr (CL) cg::this_cluster().sync();  // the others may still read this CTA's last rows
}
template <typename T>
__global__ void __launch_bounds__(kCoopThreads, 1)
    k_panel_coop(T* __restrict__ A, int64_t n, int64_t k0, int64_t k1, int R, int32_t* __restrict__ piv,
                 int* __restrict__ info, int* __restrict__ tmo, CoopScratch<T>* cs, unsigned int bar_base,
                 long long limit) {
    panel<T, false>(A, n, k0, k1, R, piv, info, tmo, cs, bar_base, limit);
}
template <typename T>
__global__ void __launch_bounds__(kCoopThreads, 1)
    k_panel_cluster(T* __restrict__ A, int64_t n, int64_t k0, int64_t k1, int R, int32_t* __restrict__ piv,
                    int* __restrict__ info, CoopScratch<T>* cs) {
    panel<T, true>(A, n, k0, k1, R, piv, info, nullptr, cs, 0, 0);
}
// rows a CTA of the cluster takes at most: above, the update of one CTA's rows takes longer than the grid
// barrier that the cluster saves
template <typename T>
constexpr int64_t kClusterRows = sizeof(T) == 8 ? 96 : 256;

// The row swaps of panel rows [k0, k1) (LAPACK order: row r with piv[r]) composed into one
// permutation of the rows they touch (at most 2 (k1 - k0)): perm[0] = number of moved rows, then
// (dst, src) pairs: row dst holds afterwards what row src held before.  A pivot outside [r, n) is a row no
// panel wrote (its panel gave up a bounded wait) and is skipped, as in the swaps themselves.
// Each of 128 threads follows one touched row's content through the swaps: thread t < 64 the
// panel row k0 + t, thread 64 + t the pivot row of step t below the panel, where no earlier
// step has it.  (One warp searching its list of rows once per swap took 20 us, this 3.)
constexpr int kSwapMax = 128;

__global__ void __launch_bounds__(kSwapMax) k_swap_perm(const int32_t* __restrict__ piv, int64_t n, int64_t k0,
                                                        int64_t k1, int32_t* __restrict__ perm) {
    __shared__ int64_t pv[kSwapMax / 2];
    __shared__ int s_cnt;
    const int w = (int)(k1 - k0), t = threadIdx.x;
    if (t == 0) s_cnt = 0;
    if (t < w) {
        const int64_t r = k0 + t, p = piv[r];
        pv[t] = (p > r && p < n) ? p : r;
    }
    __syncthreads();
    int64_t src = -1;
    if (t < w) {
        src = k0 + t;
    } else if (t >= kSwapMax / 2 && t - kSwapMax / 2 < w) {
        const int q = t - kSwapMax / 2;
        src = pv[q] >= k1 ? pv[q] : -1;
        for (int r = 0; r < q; ++r)
            if (pv[r] == src) src = -1;
    }
    int64_t at = src;
    if (src >= 0)
        for (int r = 0; r < w; ++r) {
            const int64_t p = pv[r];
            if (at == k0 + r)
                at = p;
            else if (at == p)
                at = k0 + r;
        }
    // moved rows: (dst, src) pairs after the count
    if (at != src) {
        const int c = atomicAdd(&s_cnt, 1);
        perm[1 + 2 * c] = (int32_t)at;
        perm[2 + 2 * c] = (int32_t)src;
    }
    __syncthreads();
    if (t == 0) perm[0] = s_cnt;
}

// The composed swaps applied to every column outside the panel: each thread loads all the
// moved values of its column (independent loads, staged in shared memory), then stores
// them; the result equals the swaps applied one after the other.
constexpr int kSwapThreads = 64;

template <typename T>
__global__ void __launch_bounds__(kSwapThreads) k_laswp(T* __restrict__ A, int64_t n, int64_t k0, int64_t k1,
                                                        const int32_t* __restrict__ perm) {
    extern __shared__ __align__(16) unsigned char swap_sm[];
    T* vals = reinterpret_cast<T*>(swap_sm);  // [kSwapMax][kSwapThreads]
    const int cnt = perm[0];
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n || (c >= k0 && c < k1)) return;
    T* col = A + c * n;
    // loads in batches of 16 held in registers, so that they are in flight together
    for (int i0 = 0; i0 < cnt; i0 += 16) {
        T v[16];
#pragma unroll
        for (int q = 0; q < 16; ++q)
            if (i0 + q < cnt) v[q] = col[perm[2 + 2 * (i0 + q)]];
#pragma unroll
        for (int q = 0; q < 16; ++q)
            if (i0 + q < cnt) vals[(i0 + q) * kSwapThreads + threadIdx.x] = v[q];
    }
    for (int i = 0; i < cnt; ++i) col[perm[1 + 2 * i]] = vals[i * kSwapThreads + threadIdx.x];
}

// Inverse of the unit-lower nb x nb diagonal block at (k0, k0) into W (nb x nb, ld nb), nb <= 64:
// a warp per column c, lane l holding rows l and l + 32 of it: X = e_c, then for q = c .. nb-2 (X[q]
// is final) X[r] -= L[r][q] X[q] for r > q.  The columns are independent, so nb / 8 blocks share
// the work without block barriers; one block for all, a barrier per q, took 28 us in FP32 and
// 35 us in FP64 (where one SM's FP64 pipe was the bound).
constexpr int kTriWarps = 8;

template <typename T>
__global__ void __launch_bounds__(32 * kTriWarps) k_trtri_unit_lower(const T* __restrict__ A, int64_t n, int64_t k0,
                                                                    int nb, T* __restrict__ W) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int ld = nb + 1;
    T* L = reinterpret_cast<T*>(smem_raw);  // nb x (nb+1), column q at L + q ld
    for (int idx = threadIdx.x; idx < nb * nb; idx += blockDim.x) {
        const int r = idx % nb, q = idx / nb;
        L[r + q * ld] = A[(k0 + r) + (k0 + q) * n];
    }
    __syncthreads();
    const int c = blockIdx.x * kTriWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (c >= nb) return;
    T x0 = lane == c ? (T)1 : (T)0, x1 = lane + 32 == c ? (T)1 : (T)0;
    for (int q = c; q + 1 < nb; ++q) {
        const T xq = __shfl_sync(0xffffffffu, q < 32 ? x0 : x1, q & 31);
        if (lane > q && lane < nb) x0 -= L[lane + q * ld] * xq;
        if (lane + 32 > q && lane + 32 < nb) x1 -= L[lane + 32 + q * ld] * xq;
    }
    if (lane < nb) W[lane + (int64_t)c * nb] = x0;
    if (lane + 32 < nb) W[lane + 32 + (int64_t)c * nb] = x1;
}

// U12 of a block row: X = L^-1 A[K0 : K0 + 64 nbk, c0 : c1] for the unit-lower L of nbk
// diagonal 64-blocks at (K0, K0), by block forward substitution
//   X_i = Linv_i (A_i - sum_{j < i} L_ij X_j),
// with Linv_i (nbk blocks of 64 x 64, ld 64) from k_trtri_unit_lower and L_ij read from A.
// One CTA per kTrsmCols columns holds its tile of the block row in shared memory (all nbk
// blocks), staging one 64 x 64 block of L (or Linv) at a time; thread t owns row t % 64 and
// kTrsmPer columns of the current 64-row block.  Dynamic shared memory:
// trsm_block_smem<T>(nbk).
// FP64 takes 8 columns per CTA: 64 x 64 x 8 products already hold one SM's FP64 pipe for 8 us, and
// 32 columns left most SMs idle (43 us a block row at n = 6145, 36 at 384; 8 columns: 23 and 10).
template <typename T>
constexpr int kTrsmPer = sizeof(T) == 8 ? 2 : 8;  // columns per thread
template <typename T>
constexpr int kTrsmCols = 4 * kTrsmPer<T>;

template <typename T>
__host__ __device__ constexpr size_t trsm_block_smem(int nbk) {
    return sizeof(T) * ((size_t)64 * nbk * (kTrsmCols<T> + 1) + (size_t)64 * 65);
}

template <typename T>
__global__ void __launch_bounds__(256) k_trsm_block(T* __restrict__ A, int64_t n, int64_t K0, int nbk,
                                                    const T* __restrict__ Linv, int64_t c0, int64_t c1) {
    constexpr int kP = kTrsmPer<T>, kC = kTrsmCols<T>;
    extern __shared__ __align__(16) unsigned char trsm_blk_sm[];
    T(*X)[kC + 1] = reinterpret_cast<T(*)[kC + 1]>(trsm_blk_sm);
    T(*L)[65] = reinterpret_cast<T(*)[65]>(trsm_blk_sm + sizeof(T) * 64 * nbk * (kC + 1));
    const int64_t cb = c0 + (int64_t)blockIdx.x * kC;
    const int wc = (int)min((int64_t)kC, c1 - cb);
    const int rows = 64 * nbk;
    const int r = threadIdx.x % 64, g = threadIdx.x / 64;
    for (int idx = threadIdx.x; idx < rows * kC; idx += 256) {
        const int rr = idx % rows, cc = idx / rows;
        X[rr][cc] = cc < wc ? A[(K0 + rr) + (cb + cc) * n] : (T)0;
    }
    T acc[kP];
    for (int i = 0; i < nbk; ++i) {
        // X_i -= L_ij X_j, j < i
        for (int j = 0; j < i; ++j) {
            __syncthreads();
            for (int idx = threadIdx.x; idx < 64 * 64; idx += 256) {
                const int rr = idx % 64, q = idx / 64;
                L[rr][q] = A[(K0 + 64 * i + rr) + (K0 + 64 * j + q) * n];
            }
            __syncthreads();
#pragma unroll
            for (int c = 0; c < kP; ++c) acc[c] = (T)0;
            for (int q = 0; q < 64; ++q) {
                const T l = L[r][q];
#pragma unroll
                for (int c = 0; c < kP; ++c) acc[c] = fma(l, X[64 * j + q][kP * g + c], acc[c]);
            }
#pragma unroll
            for (int c = 0; c < kP; ++c) X[64 * i + r][kP * g + c] -= acc[c];
        }
        // X_i = Linv_i X_i
        __syncthreads();
        for (int idx = threadIdx.x; idx < 64 * 64; idx += 256) {
            const int rr = idx % 64, q = idx / 64;
            L[rr][q] = Linv[(size_t)i * 64 * 64 + rr + q * 64];
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < kP; ++c) acc[c] = (T)0;
        for (int q = 0; q <= (r | 31); ++q) {  // Linv is lower triangular: the warp's last row
            const T l = L[r][q];
#pragma unroll
            for (int c = 0; c < kP; ++c) acc[c] = fma(l, X[64 * i + q][kP * g + c], acc[c]);
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < kP; ++c) X[64 * i + r][kP * g + c] = acc[c];
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < rows * kC; idx += 256) {
        const int rr = idx % rows, cc = idx / rows;
        if (cc < wc) A[(K0 + rr) + (cb + cc) * n] = X[rr][cc];
    }
}

// C = alpha * A * B + beta * C; column-major, M x N x K; 64 x 64 tiles, 256 threads, 4x4
// register tile per thread.
template <typename T>
__global__ void __launch_bounds__(256) k_gemm(int64_t M, int64_t N, int64_t K, T alpha, const T* __restrict__ A,
                                              int64_t lda, const T* __restrict__ B, int64_t ldb, T beta,
                                              T* __restrict__ C, int64_t ldc) {
    constexpr int BM = 64, BN = 64, BK = 16;
    __shared__ T As[BK][BM + 1];
    __shared__ T Bs[BK][BN + 1];
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    const int64_t m0 = (int64_t)blockIdx.x * BM, n0 = (int64_t)blockIdx.y * BN;
    T acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = (T)0;
    for (int64_t k0 = 0; k0 < K; k0 += BK) {
        for (int idx = threadIdx.x; idx < BM * BK; idx += 256) {
            const int r = idx % BM, kk = idx / BM;
            const int64_t gr = m0 + r, gk = k0 + kk;
            As[kk][r] = (gr < M && gk < K) ? A[gr + gk * lda] : (T)0;
        }
        for (int idx = threadIdx.x; idx < BN * BK; idx += 256) {
            const int kk = idx % BK, c = idx / BK;
            const int64_t gk = k0 + kk, gc = n0 + c;
            Bs[kk][c] = (gk < K && gc < N) ? B[gk + gc * ldb] : (T)0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            T a[4], b[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                a[q] = As[kk][tx + 16 * q];
                b[q] = Bs[kk][ty + 16 * q];
            }
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[p][q] = fma(a[p], b[q], acc[p][q]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t gr = m0 + tx + 16 * p, gc = n0 + ty + 16 * q;
            if (gr < M && gc < N) {
                T* c = C + gr + gc * ldc;
                *c = (beta == (T)0) ? alpha * acc[p][q] : fma(alpha, acc[p][q], beta * *c);
            }
        }
}

template <typename T>
__global__ void k_copy_block(const T* __restrict__ W, int64_t ldw, T* __restrict__ A, int64_t lda, int64_t rows,
                             int64_t cols) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= rows * cols) return;
    const int64_t r = t % rows, c = t / rows;
    A[r + c * lda] = W[r + c * ldw];
}

template <typename T>
cudaError_t gemm(int64_t M, int64_t N, int64_t K, T alpha, const T* A, int64_t lda, const T* B, int64_t ldb, T beta,
                 T* C, int64_t ldc, cudaStream_t s) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    dim3 grid((unsigned)((M + 63) / 64), (unsigned)((N + 63) / 64));
    k_gemm<T><<<grid, 256, 0, s>>>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc);
    return cudaGetLastError();
}

#define NB_TRY(x)                              \
    do {                                       \
        cudaError_t e_ = (x);                  \
        if (e_ != cudaSuccess) return e_;      \
    } while (0)

constexpr int kSuperPanels = 4;  // panels per super-panel of the two-level FP32 factorisation

// The stream on which the FP64 factorisation takes the next panel while the rest of the trailing
// update runs.  A panel is bound by latency and leaves the SMs nearly idle: with the update of the
// panel's columns first, the panel then beside the other columns' update (its CTAs at the higher priority,
// beside the update's in registers and shared memory up to 8,000 rows), the LU of 6,145 rows takes 40.2 ms
// instead of 44.4 (8,192: 65.0 and 72.6, 12,000: 151 and 164; with an update by 36 digit products).  The two share the FP64 pipe: beside the
// update a panel takes 310 us instead of 206.  Where kAheadFrom rows or more are left: below, the second
// update launch and the events cost more (1,024 rows: 4.00 and 3.88 ms; 2,500: 11.5 and 11.4; 3,000: 14.1 and 14.3).
constexpr int64_t kAheadFrom = 2048;
struct Ahead {
    cudaStream_t stream = nullptr;
    cudaEvent_t ready = nullptr, done = nullptr;
    cudaError_t init() {
        int lo = 0, hi = 0;
        cudaError_t e = cudaDeviceGetStreamPriorityRange(&lo, &hi);
        if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&stream, cudaStreamNonBlocking, hi);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ready, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&done, cudaEventDisableTiming);
        return e;
    }
    bool joined = true;  // the caller's stream waits for all that was queued here
    ~Ahead() {
        if (!joined) cudaStreamSynchronize(stream);
        if (done) cudaEventDestroy(done);
        if (ready) cudaEventDestroy(ready);
        if (stream) cudaStreamDestroy(stream);
    }
};

// work layout: [0, 4 nb*nb) unit-lower inverses; then nb*n U12 staging; then kPivBlocks doubles + kPivBlocks
// int64 for the pivot search, one int ticket and the composed row swaps.
template <typename T>
cudaError_t lu_factor(T* A, int64_t n, int32_t* piv, int nb, T* work, int* d_info, void* split, void* coop,
                      cudaStream_t s, long long polls) {
    // d_info[0]: first zero pivot (1-based) or 0; d_info[1]: a bounded wait gave up (the
    // tensor-core update or the cooperative panel's barrier); polls > 0: the barrier's
    // poll limit (default kCoopSpinLimit)
    NB_TRY(cudaMemsetAsync(d_info, 0, 2 * sizeof(int), s));
    T* Linv = work;                                         // kSuperPanels unit-lower inverses
    T* W = work + (size_t)kSuperPanels * nb * nb;
    char* tail = reinterpret_cast<char*>(W + (size_t)nb * n);
    size_t off = ((uintptr_t)tail + 15) & ~(uintptr_t)15;
    double* pval = reinterpret_cast<double*>(off);
    int64_t* pidx = reinterpret_cast<int64_t*>(pval + kPivBlocks);
    int* ticket = reinterpret_cast<int*>(pidx + kPivBlocks);
    int32_t* swap_perm = reinterpret_cast<int32_t*>(ticket + 4);  // 1 + 2 kSwapMax ints
    NB_TRY(cudaMemsetAsync(ticket, 0, sizeof(int), s));
    const int swap_smem = (int)(sizeof(T) * kSwapMax * kSwapThreads);
    NB_TRY(cudaFuncSetAttribute(k_laswp<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, swap_smem));
    if (nb > 64) return cudaErrorInvalidValue;  // k_panel_col stages at most 64 row values
    // the whole panel in one cooperative launch when every CTA's rows fit in shared
    // memory (R rows x 64 columns, R = max(kCoopMinRows, rows / SMs)) and all CTAs can be resident
    int gmax = 0;
    CoopScratch<T>* cs = static_cast<CoopScratch<T>*>(coop);
    if (cs) {
        int dev = 0, sms = 0, can = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&can, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && can) {
            const int g = std::min(kCoopMaxG, sms);
            const int64_t R0 = std::max<int64_t>(kCoopMinRows<T>, (n + g - 1) / g);
            const int64_t smem0 = R0 * 64 * (int64_t)sizeof(T);
            int per_sm = 0;
            if (smem0 <= kCoopSmemMax &&
                cudaFuncSetAttribute(k_panel_coop<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kCoopSmemMax) ==
                    cudaSuccess &&
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_panel_coop<T>, kCoopThreads, (size_t)smem0) ==
                    cudaSuccess &&
                per_sm >= 1) {
                // beside another kernel's CTA on an SM (Ahead) only if the SM's carve-out has room for both
                NB_TRY(cudaFuncSetAttribute(k_panel_coop<T>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                            cudaSharedmemCarveoutMaxShared));
                gmax = g;
                NB_TRY(cudaMemsetAsync(cs, 0, sizeof(CoopScratch<T>), s));
            }
        }
        cudaGetLastError();  // a refused attribute or query leaves the per-column path
    }
    // panels of few rows in one cluster, where the device can hold it
    cudaLaunchAttribute cl_attr{};
    cl_attr.id = cudaLaunchAttributeClusterDimension;
    cl_attr.val.clusterDim = {kPanelCluster, 1, 1};
    cudaLaunchConfig_t cl{};
    cl.gridDim = dim3(kPanelCluster);
    cl.blockDim = dim3(kCoopThreads);
    cl.dynamicSmemBytes = (size_t)kClusterRows<T> * 64 * sizeof(T);
    cl.stream = s;
    cl.attrs = &cl_attr;
    cl.numAttrs = 1;
    int clusters = 0;
    if (gmax > 0 &&
        (cudaFuncSetAttribute(k_panel_cluster<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
         cudaFuncSetAttribute(k_panel_cluster<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)cl.dynamicSmemBytes) != cudaSuccess ||
         cudaFuncSetAttribute(k_panel_cluster<T>, cudaFuncAttributePreferredSharedMemoryCarveout,
                              cudaSharedmemCarveoutMaxShared) != cudaSuccess ||
         cudaOccupancyMaxActiveClusters(&clusters, k_panel_cluster<T>, &cl) != cudaSuccess)) {
        clusters = 0;
        cudaGetLastError();
    }
    unsigned int arrivals = 0;
    // FP32 with the bulk tensor-core path: two-level blocking.  Super-panels of kSuperPanels
    // panels; inside one, each panel's U12 and update stop at the super-panel's last column;
    // after it, the block row's U12 by block forward substitution and one trailing update of
    // depth kSuperPanels * nb, so C is read and written once per super-panel.
    bool super = false;
    if constexpr (sizeof(T) == 4) super = split && nb == 64 && (n % 4) == 0 && n > (int64_t)kSuperPanels * nb;
    const int64_t sp = super ? (int64_t)kSuperPanels * nb : (int64_t)nb;
    auto trsm_rows = [&](int64_t r0, int wr, int64_t c0, int64_t c1) -> cudaError_t {
        // A[r0 : r0 + wr, c0 : c1] = L(r0 block)^-1 A[r0 : r0 + wr, c0 : c1] (unit lower wr x wr)
        const int64_t m = c1 - c0;
        k_trtri_unit_lower<T><<<(unsigned)((wr + kTriWarps - 1) / kTriWarps), 32 * kTriWarps,
                                sizeof(T) * wr * (wr + 1), s>>>(A, n, r0, wr, Linv);
        NB_TRY(gemm<T>(wr, m, wr, (T)1, Linv, wr, A + r0 + c0 * n, n, (T)0, W, wr, s));
        k_copy_block<T><<<(unsigned)((wr * m + 255) / 256), 256, 0, s>>>(W, wr, A + r0 + c0 * n, n, wr, m);
        return cudaGetLastError();
    };
    auto trsm_block = [&](int64_t r0, int nbk, const T* inv, int64_t c0, int64_t c1) -> cudaError_t {
        const int smem = (int)trsm_block_smem<T>(nbk);
        NB_TRY(cudaFuncSetAttribute(k_trsm_block<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)trsm_block_smem<T>(kSuperPanels)));
        k_trsm_block<T><<<(unsigned)((c1 - c0 + kTrsmCols<T> - 1) / kTrsmCols<T>), 256, smem, s>>>(A, n, r0, nbk, inv,
                                                                                                  c0, c1);
        return cudaGetLastError();
    };
    // the panel [k0, k1) and the permutation of its swaps, on stream st
    auto panel_step = [&](int64_t k0, int64_t k1, cudaStream_t st) -> cudaError_t {
        const int w = (int)(k1 - k0);
        if (clusters > 0 && n - k0 <= kClusterRows<T> * kPanelCluster) {
            const int R = (int)((n - k0 + kPanelCluster - 1) / kPanelCluster);
            cl.dynamicSmemBytes = (size_t)R * w * sizeof(T);
            cl.stream = st;
            NB_TRY(cudaLaunchKernelEx(&cl, k_panel_cluster<T>, A, n, k0, k1, R, piv, d_info, cs));
        } else if (gmax > 0) {
            const int64_t rows = n - k0;
            const int R = (int)std::max<int64_t>(kCoopMinRows<T>, (rows + gmax - 1) / gmax);
            const int G = (int)((rows + R - 1) / R);
            T* Af = A;
            int64_t nn = n, kk0 = k0, kk1 = k1;
            int RR = R;
            int* tmo = d_info + 1;
            unsigned int base = arrivals;
            arrivals += (unsigned int)G * (unsigned int)w;
            long long lim = polls > 0 ? polls : kCoopSpinLimit;
            void* args[] = {&Af, &nn, &kk0, &kk1, &RR, &piv, &d_info, &tmo, &cs, &base, &lim};
            NB_TRY(cudaLaunchCooperativeKernel((const void*)k_panel_coop<T>, dim3((unsigned)G), dim3(kCoopThreads),
                                               args, (size_t)R * w * sizeof(T), st));
        } else {
            // columns k0..k1-1: update by the previous column + pivot of this one; then the
            // last column's scaling of the rows below the panel
            for (int64_t j = k0; j <= k1; ++j) {
                if (j == n) break;
                const int64_t rows = n - j;
                const int pb = (int)std::min<int64_t>(kPivBlocks, (rows + kPivThreads - 1) / kPivThreads);
                k_panel_col<T><<<pb, kPivThreads, 0, st>>>(A, n, j, k0, k1, j < k1 ? 1 : 0, pval, pidx, ticket,
                                                          piv, d_info);
            }
        }
        k_swap_perm<<<1, kSwapMax, 0, st>>>(piv, n, k0, k1, swap_perm);
        return cudaGetLastError();
    };
    Ahead ahead;
    const bool look = sizeof(T) == 8 && split && nb == 64 && n - nb >= kAheadFrom;
    if (look) NB_TRY(ahead.init());
    bool panel_done = false;  // taken ahead
    for (int64_t K0 = 0; K0 < n; K0 += sp) {
        const int64_t K1 = std::min<int64_t>(n, K0 + sp);
        const int64_t e1 = super ? K1 : n;  // last column (exclusive) the panels' updates reach
        for (int64_t k0 = K0; k0 < K1; k0 += nb) {
            const int64_t k1 = std::min<int64_t>(n, k0 + nb);
            const int w = (int)(k1 - k0);
            if (!panel_done) NB_TRY(panel_step(k0, k1, s));
            panel_done = false;
            k_laswp<T><<<(unsigned)((n + kSwapThreads - 1) / kSwapThreads), kSwapThreads, swap_smem, s>>>(A, n, k0,
                                                                                                    k1, swap_perm);
            const bool tc64 = sizeof(T) == 8 && split;  // FP64 with the tensor-core update
            if ((super && (k1 < K1 || K1 < n)) || (tc64 && w == 64 && k1 < n)) {
                // the panel's unit-lower inverse, kept in its slot for the block row's U12
                T* slot = Linv + (size_t)((k0 - K0) / nb) * nb * nb;
                k_trtri_unit_lower<T><<<(unsigned)((w + kTriWarps - 1) / kTriWarps), 32 * kTriWarps,
                                        sizeof(T) * w * (w + 1), s>>>(A, n, k0, w, slot);
            }
            if (k1 < e1) {
                const int64_t m = n - k1, mc = e1 - k1;
                if (super || (tc64 && w == 64))
                    NB_TRY(trsm_block(k0, 1, Linv + (size_t)((k0 - K0) / nb) * nb * nb, k1, e1));
                else
                    NB_TRY(trsm_rows(k0, w, k1, e1));
                // A22 -= L21 * U12 over the columns up to e1: tensor cores (TF32 x3) for the
                // FP32 factorisation's 64-wide panels, FP64 FMA for the FP64 factorisation
                if constexpr (sizeof(T) == 4) {
                    if (w == 64) {
                        NB_TRY(tc_update_f32(m, mc, reinterpret_cast<const float*>(A + k1 + k0 * n), n,
                                             reinterpret_cast<const float*>(A + k0 + k1 * n), n,
                                             reinterpret_cast<float*>(A + k1 + k1 * n), n, split, d_info + 1, s));
                        continue;
                    }
                } else if (tc64) {
                    const T *L21 = A + k1 + k0 * n, *U12 = A + k0 + k1 * n;
                    T* C = A + k1 + k1 * n;
                    NB_TRY(tc_split_f64(m, mc, w, L21, n, U12, n, split, s));
                    if (look && m >= kAheadFrom) {
                        NB_TRY(tc_apply_f64(m, mc, w, 0, nb, L21, n, U12, n, C, n, split, d_info + 1, s));
                        NB_TRY(cudaEventRecord(ahead.ready, s));
                        NB_TRY(cudaStreamWaitEvent(ahead.stream, ahead.ready, 0));
                        ahead.joined = false;
                        NB_TRY(panel_step(k1, k1 + nb, ahead.stream));
                        NB_TRY(cudaEventRecord(ahead.done, ahead.stream));
                        NB_TRY(tc_apply_f64(m, mc, w, nb, mc, L21, n, U12, n, C, n, split, d_info + 1, s));
                        NB_TRY(cudaStreamWaitEvent(s, ahead.done, 0));
                        ahead.joined = true;
                        panel_done = true;
                    } else {
                        NB_TRY(tc_apply_f64(m, mc, w, 0, mc, L21, n, U12, n, C, n, split, d_info + 1, s));
                    }
                    continue;
                }
                NB_TRY(gemm<T>(m, mc, w, (T)-1, A + k1 + k0 * n, n, A + k0 + k1 * n, n, (T)1, A + k1 + k1 * n, n, s));
            }
            NB_TRY(cudaGetLastError());
        }
        if constexpr (sizeof(T) == 4) {
            if (super && K1 < n) {
                const int64_t m = n - K1;
                // U12 of the block row [K0, K1) over the trailing columns: block forward
                // substitution with the super-panel's unit-lower blocks and their inverses
                NB_TRY(trsm_block(K0, kSuperPanels, Linv, K1, n));
                NB_TRY(tc_update_f32_k(m, m, K1 - K0, reinterpret_cast<const float*>(A + K1 + K0 * n), n,
                                       reinterpret_cast<const float*>(A + K0 + K1 * n), n,
                                       reinterpret_cast<float*>(A + K1 + K1 * n), n, split, d_info + 1, s));
            }
        }
    }
    return cudaSuccess;
}

// ---------------------------------------------------------------- triangular solves
constexpr int kTB = 64;          // solve block
constexpr int kResRows = 256;    // residual: rows per CTA
constexpr int kResChunk = 512;   // residual: columns per partial sum (enough (row, chunk) threads to keep HBM busy)

// Row permutation of the pivots: applying the swaps (k, piv[k]), k = 0..n-1, to b gives
// b'[i] = b[perm[i]].  The swaps are sequential; they run on an index array in shared
// memory (one thread) when it fits, else in global memory.
__global__ void k_make_perm_smem(const int32_t* __restrict__ piv, int64_t n, int32_t* __restrict__ perm) {
    extern __shared__ int32_t sp[];
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) sp[i] = (int32_t)i;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int64_t k = 0; k < n; ++k) {
            const int32_t p = (piv[k] >= k && piv[k] < n) ? piv[k] : (int32_t)k;  // caller pivots: stay in range
            if (p != k) {
                const int32_t t = sp[k];
                sp[k] = sp[p];
                sp[p] = t;
            }
        }
    }
    __syncthreads();
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) perm[i] = sp[i];
}

__global__ void k_make_perm_global(const int32_t* __restrict__ piv, int64_t n, int32_t* __restrict__ perm) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    for (int64_t i = 0; i < n; ++i) perm[i] = (int32_t)i;
    for (int64_t k = 0; k < n; ++k) {
        const int32_t p = (piv[k] >= k && piv[k] < n) ? piv[k] : (int32_t)k;
        if (p != k) {
            const int32_t t = perm[k];
            perm[k] = perm[p];
            perm[p] = t;
        }
    }
}

// Values that CTAs of one launch pass to one another through memory are their own flags: the array is
// filled with the pattern of all ones (a NaN that no operation produces) and read with relaxed
// loads until another value is there.
__device__ __forceinline__ void ld_passed(const float* p, float& v, bool& set) {
    uint32_t u;
    asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(u) : "l"(p) : "memory");
    v = __uint_as_float(u);
    set = u != 0xffffffffu;
}
__device__ __forceinline__ void ld_passed(const double* p, double& v, bool& set) {
    unsigned long long u;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(u) : "l"(p) : "memory");
    v = __longlong_as_double((long long)u);
    set = u != ~0ull;
}
__device__ __forceinline__ void st_passed(float* p, float v) {
    if (v != v) v = __uint_as_float(0x7fc00000u);
    asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(__float_as_uint(v)) : "memory");
}
__device__ __forceinline__ void st_passed(double* p, double v) {
    if (v != v) v = __longlong_as_double(0x7ff8000000000000ll);
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(__double_as_longlong(v)) : "memory");
}
__device__ __forceinline__ void set_unpassed(float& v) { v = __uint_as_float(0xffffffffu); }
__device__ __forceinline__ void set_unpassed(double& v) { v = __longlong_as_double(-1ll); }

// y = b permuted; z is made ready for the lower sweep's values
template <typename T>
__global__ void k_permute(const T* __restrict__ b, const int32_t* __restrict__ perm, int64_t n, T* __restrict__ y,
                          T* __restrict__ z) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    y[i] = b[perm[i]];
    set_unpassed(z[i]);
}

// One triangular sweep in one launch.  Block rows of kTB rows; the CTA with ticket t (taken
// from an atomic counter, so tickets follow the order in which CTAs start) solves block k =
// t (lower sweep, unit-diagonal L) or nblk-1-t (upper sweep, U):
//   x_k = D_k^-1 (rhs_k - sum_c M_kc x_c),  c < k (lower) or c > k (upper),
// taking the blocks c in sweep order as their solutions appear in x, which was filled with the
// pattern of ld_passed (the lower sweep fills the upper sweep's).  A CTA only waits for
// blocks of lower tickets, whose CTAs have started, so the waits end.  Each thread owns one
// row of the block and a quarter of its columns, and every warp waits for its 16 values by
// itself; the matrix values of the next block are in flight meanwhile.  The four partial sums are
// added in a fixed order, so the result does not depend on timing.
// Diagonal block: FP64 sweeps solve it by substitution in one warp (warp_substitute); FP32
// sweeps (the inner solves of the iterative refinement) invert it in shared memory while
// the CTA waits, so that the step on the critical path is a 64 x 64 matrix-vector product.
// Every wait is bounded: on giving up the CTA records *err and passes NaN for its block.
// Bound by the chain over the blocks (value to the next CTA, its product, sum and diagonal block): 64
// rows take 1.1 us in FP32 and 8.5 us in FP64 (3.1 and 15 us with flags that one thread polls
// and the block barriers around them, and with the substitution in shared memory).
constexpr int kSvThreads = 256;
constexpr long long kSvSpinLimit = 1ll << 22;

// xs = D^-1 xs for the block's w rows by one warp, two rows to a lane, the solved value broadcast
// by shuffle: L (unit diagonal) downwards, U upwards with the reciprocals of its diagonal.
// D is zero outside its w x w entries.
template <typename T>
__device__ __forceinline__ void warp_substitute(const T (*__restrict__ D)[kTB + 1], const T* __restrict__ dinv,
                                                T* xs, int w, bool lower) {
    static_assert(kTB == 64, "two rows per lane");
    const int lane = threadIdx.x % 32;
    const bool has0 = lane < w, has1 = lane + 32 < w;
    T a0 = has0 ? xs[lane] : (T)0, a1 = has1 ? xs[lane + 32] : (T)0;
    if (lower) {
        const int m = min(w, 32);
#pragma unroll 8
        for (int c = 0; c < m; ++c) {
            const T d0 = D[lane][c], d1 = D[lane + 32][c];
            const T xc = __shfl_sync(0xffffffffu, a0, c);
            if (lane > c) a0 = fma(-d0, xc, a0);
            a1 = fma(-d1, xc, a1);
        }
#pragma unroll 8
        for (int c = 32; c < w; ++c) {
            const T d1 = D[lane + 32][c];
            const T xc = __shfl_sync(0xffffffffu, a1, c - 32);
            if (lane + 32 > c) a1 = fma(-d1, xc, a1);
        }
    } else {
        const T i0 = has0 ? dinv[lane] : (T)0, i1 = has1 ? dinv[lane + 32] : (T)0;
#pragma unroll 8
        for (int c = w - 1; c >= 32; --c) {
            const T d0 = D[lane][c], d1 = D[lane + 32][c];
            const T xc = __shfl_sync(0xffffffffu, a1 * i1, c - 32);
            if (lane + 32 < c) a1 = fma(-d1, xc, a1);
            a0 = fma(-d0, xc, a0);
        }
#pragma unroll 8
        for (int c = min(w, 32) - 1; c >= 0; --c) {
            const T d0 = D[lane][c];
            const T xc = __shfl_sync(0xffffffffu, a0 * i0, c);
            if (lane < c) a0 = fma(-d0, xc, a0);
        }
        a0 *= i0;
        a1 *= i1;
    }
    if (has0) xs[lane] = a0;
    if (has1) xs[lane + 32] = a1;
}

// X = D^-1, each warp kTB / warps columns in registers (two rows to a lane), eliminated together.  (9 us
// with the columns in shared memory and a block barrier per step; every sweep starts with it.)
template <typename T>
__device__ __forceinline__ void warp_invert(const T (*__restrict__ D)[kTB + 1], const T* __restrict__ dinv,
                                            T (*__restrict__ X)[kTB + 1], int w, bool lower) {
    constexpr int kC = kTB / (kSvThreads / 32);
    const int lane = threadIdx.x % 32, c0 = threadIdx.x / 32 * kC;
    T a0[kC], a1[kC];
#pragma unroll
    for (int j = 0; j < kC; ++j) {
        a0[j] = lane == c0 + j && lane < w ? (T)1 : (T)0;
        a1[j] = lane + 32 == c0 + j && lane + 32 < w ? (T)1 : (T)0;
    }
    if (lower) {
        for (int q = 0; q + 1 < w; ++q) {
            const T d0 = D[lane][q], d1 = D[lane + 32][q];
#pragma unroll
            for (int j = 0; j < kC; ++j) {
                const T x = __shfl_sync(0xffffffffu, q < 32 ? a0[j] : a1[j], q & 31);
                if (lane > q) a0[j] = fma(-d0, x, a0[j]);
                if (lane + 32 > q) a1[j] = fma(-d1, x, a1[j]);
            }
        }
    } else {
        const T i0 = lane < w ? dinv[lane] : (T)0, i1 = lane + 32 < w ? dinv[lane + 32] : (T)0;
        for (int q = w - 1; q >= 0; --q) {
            const T d0 = D[lane][q], d1 = D[lane + 32][q], iq = dinv[q];
#pragma unroll
            for (int j = 0; j < kC; ++j) {
                const T v = __shfl_sync(0xffffffffu, q < 32 ? a0[j] : a1[j], q & 31) * iq;
                const T x = c0 + j >= q ? v : (T)0;  // X is upper triangular, also beside a zero pivot
                if (lane < q) a0[j] = fma(-d0, x, a0[j]);
                if (lane + 32 < q) a1[j] = fma(-d1, x, a1[j]);
            }
        }
#pragma unroll
        for (int j = 0; j < kC; ++j) {
            if (lane <= c0 + j) a0[j] *= i0;
            if (lane + 32 <= c0 + j) a1[j] *= i1;
        }
    }
#pragma unroll
    for (int j = 0; j < kC; ++j) {
        X[lane][c0 + j] = a0[j];
        X[lane + 32][c0 + j] = a1[j];
    }
}

template <typename T>
__global__ void __launch_bounds__(kSvThreads) k_trsv(const T* __restrict__ LU, int64_t n, int64_t nblk, int lower,
                                                     const T* __restrict__ rhs, T* x, T* __restrict__ next,
                                                     int* ticket, int* err, long long limit) {
    constexpr bool kInv = sizeof(T) == 4;  // explicit inverse of the diagonal block (FP32)
    __shared__ T D[kTB][kTB + 1];
    __shared__ T Xi[kInv ? kTB : 1][kTB + 1];
    __shared__ T part[kSvThreads / kTB][kTB];
    __shared__ T xs[kTB];
    __shared__ T dinv[kTB];
    __shared__ int s_t, s_fail;
    if (threadIdx.x == 0) {
        s_t = atomicAdd(ticket, 1);
        s_fail = 0;
    }
    __syncthreads();
    const int64_t t = s_t;
    const int64_t k = lower ? t : nblk - 1 - t;
    const int64_t r0 = k * kTB, r1 = min(n, r0 + (int64_t)kTB);
    const int w = (int)(r1 - r0);
    constexpr int kGroups = kSvThreads / kTB, kCols = kTB / kGroups;
    const int row = threadIdx.x % kTB, grp = threadIdx.x / kTB;
    if (next && threadIdx.x < w) set_unpassed(next[r0 + threadIdx.x]);
    for (int idx = threadIdx.x; idx < kTB * kTB; idx += kSvThreads) {
        const int r = idx % kTB, c = idx / kTB;
        D[r][c] = (r < w && c < w) ? LU[(r0 + r) + (r0 + c) * n] : (T)0;
    }
    // independent of the other blocks: the block's right-hand side and, for U, the
    // reciprocals of its diagonal
    const T rhs_own = (threadIdx.x < w) ? rhs[r0 + threadIdx.x] : (T)0;
    if (!lower && threadIdx.x < w) dinv[threadIdx.x] = (T)1 / LU[(r0 + threadIdx.x) + (r0 + threadIdx.x) * n];
    __syncthreads();
    if constexpr (kInv) warp_invert<T>(D, dinv, Xi, w, lower);
    T acc = (T)0;
    const int64_t total = lower ? k : nblk - 1 - k;
    const int lane = threadIdx.x % 32;
    // matrix values of block i (sweep order) for this thread: row `row`, kCols columns
    T mv[kCols];
    auto load_block = [&](int64_t i, T (&m)[kCols]) {
        const int64_t c0 = (lower ? i : nblk - 1 - i) * kTB + grp * kCols;
        const T* col = LU + (r0 + row) + c0 * n;
        const int wc = (int)min((int64_t)kCols, n - c0);
#pragma unroll
        for (int q = 0; q < kCols; ++q) m[q] = (row < w && q < wc) ? col[(int64_t)q * n] : (T)0;
    };
    if (total > 0) load_block(0, mv);
    long long spins = 0;
    // block i with the matrix values m, while those of block i + 1 arrive in nx
    auto step = [&](int64_t i, const T(&m)[kCols], T(&nx)[kCols]) {
        if (i + 1 < total) load_block(i + 1, nx);
        // the warp's kCols values of x (the last block of x may be short)
        const int64_t c0 = (lower ? i : nblk - 1 - i) * kTB + grp * kCols;
        const int q = lane % kCols;
        T v = (T)0;
        bool set = true;
        for (;;) {
            if (c0 + q < n) ld_passed(x + c0 + q, v, set);
            if (__all_sync(0xffffffffu, set) || ++spins > limit) break;
            if (i + 2 < total) __nanosleep(64);  // this block is not the next one's critical path
        }
        if (!__all_sync(0xffffffffu, set)) return false;
#pragma unroll
        for (int j = 0; j < kCols; ++j) acc = fma(m[j], __shfl_sync(0xffffffffu, v, j), acc);
        return true;
    };
    T mw[kCols];
    for (int64_t i = 0; i < total; i += 2)
        if (!step(i, mv, mw) || (i + 1 < total && !step(i + 1, mw, mv))) {
            if (lane == 0) s_fail = 1;
            break;
        }
    part[grp][row] = acc;
    __syncthreads();
    const bool ok = s_fail == 0;
    if (threadIdx.x < w) {
        T sum = part[0][threadIdx.x];
#pragma unroll
        for (int g = 1; g < kGroups; ++g) sum += part[g][threadIdx.x];
        xs[threadIdx.x] = rhs_own - sum;
    }
    __syncthreads();
    if constexpr (kInv) {
        // x = X (rhs - sum): row `row`, columns of group grp, then the groups in order
        T v = (T)0;
        if (row < w) {
#pragma unroll
            for (int q = 0; q < kCols; ++q) {
                const int c = grp * kCols + q;
                if (c < w) v = fma(Xi[row][c], xs[c], v);
            }
        }
        part[grp][row] = v;
        __syncthreads();
        if (threadIdx.x < w) {
            T sum = part[0][threadIdx.x];
#pragma unroll
            for (int g = 1; g < kGroups; ++g) sum += part[g][threadIdx.x];
            st_passed(x + r0 + threadIdx.x, ok ? sum : (T)NAN);
        }
    } else if (threadIdx.x < 32) {
        warp_substitute<T>(D, dinv, xs, w, lower);
        for (int r = threadIdx.x; r < w; r += 32) st_passed(x + r0 + r, ok ? xs[r] : (T)NAN);
    }
    if (threadIdx.x == 0 && !ok) atomicExch(err, 1);
}

// The same sweep for nr <= kMR right-hand sides at once (columns of rhs and x, leading
// dimension n; used for the weighting fields of several readouts, Sec. 2.1).  Each factor
// block is read once for all columns, and the columns share every block barrier.  Per
// column the arithmetic is k_trsv's, in its order (the fma chain over blocks and columns,
// the four group sums in order, the diagonal block: FP64 substitution, one warp per column;
// FP32 explicit inverse), so column j equals k_trsv on that column bit for bit.  Waits,
// give-up and passing as in k_trsv.  Dynamic shared memory, trsm_smem_bytes<T>():
//   D[kTB][kTB+1], Xi[kTB][kTB+1] (FP32 only), part[groups][kMR][kTB], xs[kMR][kTB] (the
//   block's right-hand sides, then its solution), dinv[kTB], xw[warps][kMR][16] (the passed values).
constexpr int kMR = 8;

template <typename T>
__host__ __device__ constexpr size_t trsm_smem_bytes() {
    return sizeof(T) * ((size_t)kTB * (kTB + 1) * (sizeof(T) == 4 ? 2 : 1) + (size_t)(kSvThreads / kTB) * kMR * kTB +
                        (size_t)kMR * kTB + kTB + (size_t)(kSvThreads / 32) * kMR * (kTB * kTB / kSvThreads));
}

template <typename T>
__global__ void __launch_bounds__(kSvThreads) k_trsm(const T* __restrict__ LU, int64_t n, int64_t nblk, int lower,
                                                     const T* __restrict__ rhs, T* x, T* __restrict__ next, int nr,
                                                     int* ticket, int* err, long long limit) {
    constexpr bool kInv = sizeof(T) == 4;
    constexpr int kGroups = kSvThreads / kTB, kCols = kTB / kGroups;
    extern __shared__ __align__(16) unsigned char trsm_sm[];
    T(*D)[kTB + 1] = reinterpret_cast<T(*)[kTB + 1]>(trsm_sm);
    T(*Xi)[kTB + 1] = D + kTB;  // FP32 only
    T(*part)[kMR][kTB] = reinterpret_cast<T(*)[kMR][kTB]>(reinterpret_cast<T*>(D + (kInv ? 2 : 1) * kTB));
    T(*xs)[kTB] = reinterpret_cast<T(*)[kTB]>(reinterpret_cast<T*>(part + kGroups));
    T* dinv = reinterpret_cast<T*>(xs + kMR);
    T(*xw)[kCols] = reinterpret_cast<T(*)[kCols]>(dinv + kTB) + kMR * (threadIdx.x / 32);
    __shared__ int s_t, s_fail;
    if (threadIdx.x == 0) {
        s_t = atomicAdd(ticket, 1);
        s_fail = 0;
    }
    __syncthreads();
    const int64_t t = s_t;
    const int64_t k = lower ? t : nblk - 1 - t;
    const int64_t r0 = k * kTB, r1 = min(n, r0 + (int64_t)kTB);
    const int w = (int)(r1 - r0);
    const int row = threadIdx.x % kTB, grp = threadIdx.x / kTB;
    for (int idx = threadIdx.x; idx < kTB * kTB; idx += kSvThreads) {
        const int r = idx % kTB, c = idx / kTB;
        D[r][c] = (r < w && c < w) ? LU[(r0 + r) + (r0 + c) * n] : (T)0;
    }
    for (int idx = threadIdx.x; idx < w * nr; idx += kSvThreads) {
        const int j = idx / w, r = idx - j * w;
        xs[j][r] = rhs[r0 + r + (int64_t)j * n];
        if (next) set_unpassed(next[r0 + r + (int64_t)j * n]);
    }
    if (!lower && threadIdx.x < w) dinv[threadIdx.x] = (T)1 / LU[(r0 + threadIdx.x) + (r0 + threadIdx.x) * n];
    __syncthreads();
    if constexpr (kInv) warp_invert<T>(D, dinv, Xi, w, lower);
    T acc[kMR];
#pragma unroll
    for (int j = 0; j < kMR; ++j) acc[j] = (T)0;
    const int64_t total = lower ? k : nblk - 1 - k;
    const int lane = threadIdx.x % 32;
    T mv[kCols];
    auto load_block = [&](int64_t i, T (&m)[kCols]) {
        const int64_t c0 = (lower ? i : nblk - 1 - i) * kTB + grp * kCols;
        const T* col = LU + (r0 + row) + c0 * n;
        const int wc = (int)min((int64_t)kCols, n - c0);
#pragma unroll
        for (int q = 0; q < kCols; ++q) m[q] = (row < w && q < wc) ? col[(int64_t)q * n] : (T)0;
    };
    if (total > 0) load_block(0, mv);
    long long spins = 0;
    auto step = [&](int64_t i, const T(&m)[kCols], T(&nx)[kCols]) {
        if (i + 1 < total) load_block(i + 1, nx);
        // the warp's kCols values of every column of x, two columns per load
        const int64_t c0 = (lower ? i : nblk - 1 - i) * kTB + grp * kCols;
        const int q = lane % kCols;
        for (int j0 = 0; j0 < nr; j0 += 32 / kCols) {
            const int j = j0 + lane / kCols;
            T v = (T)0;
            bool set = true;
            const bool mine = j < nr && c0 + q < n;
            for (;;) {
                if (mine) ld_passed(x + c0 + q + (int64_t)j * n, v, set);
                if (__all_sync(0xffffffffu, set) || ++spins > limit) break;
                if (i + 2 < total) __nanosleep(64);
            }
            if (!__all_sync(0xffffffffu, set)) return false;
            xw[j][q] = v;
        }
        __syncwarp();
#pragma unroll
        for (int c = 0; c < kCols; ++c)
#pragma unroll
            for (int j = 0; j < kMR; ++j)
                if (j < nr) acc[j] = fma(m[c], xw[j][c], acc[j]);
        __syncwarp();
        return true;
    };
    T mw[kCols];
    for (int64_t i = 0; i < total; i += 2)
        if (!step(i, mv, mw) || (i + 1 < total && !step(i + 1, mw, mv))) {
            if (lane == 0) s_fail = 1;
            break;
        }
    // every column's four group sums, in order, subtracted from its right-hand side
#pragma unroll
    for (int j = 0; j < kMR; ++j)
        if (j < nr) part[grp][j][row] = acc[j];
    __syncthreads();
    const bool ok = s_fail == 0;
    for (int idx = threadIdx.x; idx < w * nr; idx += kSvThreads) {
        const int j = idx / w, r = idx - j * w;
        T sum = part[0][j][r];
#pragma unroll
        for (int g = 1; g < kGroups; ++g) sum += part[g][j][r];
        xs[j][r] = xs[j][r] - sum;
    }
    __syncthreads();
    if constexpr (kInv) {
        // x_j = X (rhs_j - sum_j): row `row`, columns of group grp, then the groups in order
        T v[kMR];
#pragma unroll
        for (int j = 0; j < kMR; ++j) {
            v[j] = (T)0;
            if (j < nr && row < w) {
#pragma unroll
                for (int q = 0; q < kCols; ++q) {
                    const int c = grp * kCols + q;
                    if (c < w) v[j] = fma(Xi[row][c], xs[j][c], v[j]);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < kMR; ++j)
            if (j < nr) part[grp][j][row] = v[j];
        __syncthreads();
        for (int idx = threadIdx.x; idx < w * nr; idx += kSvThreads) {
            const int j = idx / w, r = idx - j * w;
            T sum = part[0][j][r];
#pragma unroll
            for (int g = 1; g < kGroups; ++g) sum += part[g][j][r];
            st_passed(x + r0 + r + (int64_t)j * n, ok ? sum : (T)NAN);
        }
    } else {
        const int j = threadIdx.x / 32;
        if (j < nr) {
            warp_substitute<T>(D, dinv, xs[j], w, lower);
            for (int r = lane; r < w; r += 32) st_passed(x + r0 + r + (int64_t)j * n, ok ? xs[j][r] : (T)NAN);
        }
    }
    if (threadIdx.x == 0 && !ok) atomicExch(err, 1);
}

template <typename T>
__global__ void k_permute_m(const T* __restrict__ b, const int32_t* __restrict__ perm, int64_t n, int nr,
                            T* __restrict__ y, T* __restrict__ z) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * nr) return;
    const int64_t j = idx / n, i = idx - j * n;
    y[idx] = b[perm[i] + j * n];
    set_unpassed(z[idx]);
}

template <typename T>
cudaError_t lu_solve(const T* LU, int64_t n, const int32_t* perm, T* b, T* work, cudaStream_t s, long long polls) {
    if (n == 0) return cudaSuccess;
    const int64_t nblk = (n + kTB - 1) / kTB;
    T* y = work;
    T* z = work + n;
    // both sweeps' tickets and the error flag (16-byte aligned after z)
    int* tickets = reinterpret_cast<int*>(((uintptr_t)(z + n) + 15) & ~(uintptr_t)15);
    int* err = tickets + 2;
    NB_TRY(cudaMemsetAsync(tickets, 0, 3 * sizeof(int), s));
    const unsigned g = (unsigned)((n + 255) / 256);
    k_permute<T><<<g, 256, 0, s>>>(b, perm, n, y, z);
    const long long limit = polls > 0 ? polls : kSvSpinLimit;
    k_trsv<T><<<(unsigned)nblk, kSvThreads, 0, s>>>(LU, n, nblk, 1, y, z, b, tickets, err, limit);
    k_trsv<T><<<(unsigned)nblk, kSvThreads, 0, s>>>(LU, n, nblk, 0, z, b, nullptr, tickets + 1, err, limit);
    return cudaGetLastError();
}

// r = b - K x for column-major K: partial sums over column chunks of kResChunk (one CTA per
// rows x chunk), then the chunks added in order per row.
__global__ void __launch_bounds__(kResRows) k_residual_partial(const double* __restrict__ K, int64_t n,
                                                               const double* __restrict__ x,
                                                               double* __restrict__ part) {
    const int64_t i = (int64_t)blockIdx.x * kResRows + threadIdx.x;
    const int64_t j0 = (int64_t)blockIdx.y * kResChunk, j1 = min(n, j0 + (int64_t)kResChunk);
    __shared__ double xs[kResChunk];
    for (int64_t j = j0 + threadIdx.x; j < j1; j += kResRows) xs[j - j0] = x[j];
    __syncthreads();
    if (i >= n) return;
    double s = 0.0;
#pragma unroll 8
    for (int64_t j = j0; j < j1; ++j) s = fma(K[i + j * n], xs[j - j0], s);
    part[(int64_t)blockIdx.y * n + i] = s;
}

__global__ void k_residual_final(const double* __restrict__ part, int64_t nchunk, int64_t n,
                                 const double* __restrict__ b, double* __restrict__ r) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double s = 0.0;
    for (int64_t c = 0; c < nchunk; ++c) s += part[c * n + i];
    r[i] = b[i] - s;
}

// r_j = b_j - K x_j for nr <= kMR columns at once (leading dimension n): K is read once for
// all columns; per column the sums are k_residual_partial's (an fma chain over the chunk's
// columns in order) and k_residual_final's (the chunks in order), so column j equals the
// single-column residual bit for bit.  x is staged in shared memory kResTile columns at a time.
constexpr int kResTile = 512;

template <int NR>
__global__ void __launch_bounds__(kResRows) k_residual_partial_m(const double* __restrict__ K, int64_t n,
                                                                 const double* __restrict__ x,
                                                                 double* __restrict__ part) {
    const int64_t i = (int64_t)blockIdx.x * kResRows + threadIdx.x;
    const int64_t j0 = (int64_t)blockIdx.y * kResChunk, j1 = min(n, j0 + (int64_t)kResChunk);
    constexpr int kUnroll = NR > 4 ? 4 : 8;  // loads in flight, within the register budget
    __shared__ double xs[kResTile][NR];
    double s[NR];
#pragma unroll
    for (int c = 0; c < NR; ++c) s[c] = 0.0;
    for (int64_t t0 = j0; t0 < j1; t0 += kResTile) {
        const int64_t t1 = min(j1, t0 + (int64_t)kResTile);
        __syncthreads();
        for (int64_t idx = threadIdx.x; idx < (t1 - t0) * NR; idx += kResRows) {
            const int64_t c = idx / (t1 - t0), j = idx - c * (t1 - t0);
            xs[j][c] = x[t0 + j + c * n];
        }
        __syncthreads();
        if (i < n)
#pragma unroll kUnroll
            for (int64_t j = t0; j < t1; ++j) {
                const double kv = K[i + j * n];
#pragma unroll
                for (int c = 0; c < NR; ++c) s[c] = fma(kv, xs[j - t0][c], s[c]);
            }
    }
    if (i < n)
#pragma unroll
        for (int c = 0; c < NR; ++c) part[((int64_t)blockIdx.y * kMR + c) * n + i] = s[c];
}

template <int NR>
static void launch_residual_partial_m(dim3 grid, cudaStream_t s, const double* K, int64_t n, const double* x,
                                      double* part) {
    k_residual_partial_m<NR><<<grid, kResRows, 0, s>>>(K, n, x, part);
}

__global__ void k_residual_final_m(const double* __restrict__ part, int64_t nchunk, int64_t n, int nr,
                                   const double* __restrict__ b, double* __restrict__ r) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * nr) return;
    const int64_t c = idx / n, i = idx - c * n;
    double s = 0.0;
    for (int64_t q = 0; q < nchunk; ++q) s += part[(q * kMR + c) * n + i];
    r[idx] = b[idx] - s;
}

// x_j += d_j for the columns j whose bit is set in `active`; norms[2j] = max|d_j|,
// norms[2j + 1] = max|x_j| (as k_ir_update, one column per blockIdx.y).
__global__ void k_ir_update_m(double* __restrict__ x, const float* __restrict__ d, int64_t n, uint32_t active,
                              double* norms) {
    const int64_t c = blockIdx.y;
    if (!((active >> c) & 1u)) return;
    double md = 0.0, mx = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double di = (double)d[i + c * n];
        const double xi = x[i + c * n] + di;
        x[i + c * n] = xi;
        md = fmax(md, fabs(di));
        mx = fmax(mx, fabs(xi));
    }
    for (int o = 16; o > 0; o >>= 1) {
        md = fmax(md, __shfl_xor_sync(0xffffffffu, md, o));
        mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(reinterpret_cast<unsigned long long*>(norms + 2 * c), __double_as_longlong(md));
        atomicMax(reinterpret_cast<unsigned long long*>(norms + 2 * c + 1), __double_as_longlong(mx));
    }
}

__global__ void k_f64_to_f32(const double* __restrict__ a, float* __restrict__ b, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        b[i] = (float)a[i];
}

// x += d; norms[0] = max|d|, norms[1] = max|x| (atomicMax on the bit patterns of
// non-negative doubles, which order like the values).
__global__ void k_ir_update(double* __restrict__ x, const float* __restrict__ d, int64_t n, double* norms) {
    double md = 0.0, mx = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double di = (double)d[i];
        const double xi = x[i] + di;
        x[i] = xi;
        md = fmax(md, fabs(di));
        mx = fmax(mx, fabs(xi));
    }
    for (int o = 16; o > 0; o >>= 1) {
        md = fmax(md, __shfl_xor_sync(0xffffffffu, md, o));
        mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(reinterpret_cast<unsigned long long*>(norms), __double_as_longlong(md));
        atomicMax(reinterpret_cast<unsigned long long*>(norms + 1), __double_as_longlong(mx));
    }
}

__global__ void k_absmax(const double* __restrict__ a, int64_t n, double* out) {
    double m = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        m = fmax(m, fabs(a[i]));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<unsigned long long*>(out), __double_as_longlong(m));
}

__global__ void k_gather(const double* __restrict__ a, const int64_t* __restrict__ idx, int64_t n,
                         double* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = a[idx[i]];
}

}  // namespace

cudaError_t launch_gather(const double* a, const int64_t* idx, int64_t n, double* out, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_gather<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, idx, n, out);
    return cudaGetLastError();
}

size_t lu_work_elems(int64_t n, int nb) {
    // L11^-1 + U12 staging + pivot partials, the ticket and the composed row swaps (in
    // 4-byte units rounded up, which covers both types)
    return (size_t)kSuperPanels * nb * nb + (size_t)nb * (size_t)n + 16 + (size_t)kPivBlocks * 4 + 16 +
           (2 * kSwapMax + 16);
}

cudaError_t lu_factor_f64_small(double* A, int64_t n, int32_t* piv, int nb, double* work, int* d_info,
                                cudaStream_t s) {
    return lu_factor<double>(A, n, piv, nb, work, d_info, nullptr, nullptr, s, 0);
}
static size_t digits_offset(int64_t n, int nb) { return (sizeof(double) * lu_work_elems(n, nb) + 255) & ~(size_t)255; }
static size_t coop64_offset(int64_t n, int nb) {
    return (digits_offset(n, nb) + tc64_work_bytes(n, n) + 255) & ~(size_t)255;
}
size_t lu_work_bytes_f64(int64_t n, int nb) { return coop64_offset(n, nb) + sizeof(CoopScratch<double>); }
cudaError_t lu_factor_f64(double* A, int64_t n, int32_t* piv, int nb, void* work, int* d_info, cudaStream_t s,
                          long long polls) {
    // work: panel staging, then the digits of the tensor-core update, then the cooperative
    // panel's candidates and barrier
    char* w = static_cast<char*>(work);
    return lu_factor<double>(A, n, piv, nb, reinterpret_cast<double*>(w), d_info, w + digits_offset(n, nb),
                             w + coop64_offset(n, nb), s, polls);
}
static size_t split_offset(int64_t n, int nb) { return (sizeof(float) * lu_work_elems(n, nb) + 255) & ~(size_t)255; }
static size_t coop_offset(int64_t n, int nb) {
    return (split_offset(n, nb) + tc_split_bytes(n, n, kSuperPanels) + 255) & ~(size_t)255;
}
size_t lu_work_bytes_f32(int64_t n, int nb) { return coop_offset(n, nb) + sizeof(CoopScratch<float>); }
cudaError_t lu_factor_f32(float* A, int64_t n, int32_t* piv, int nb, float* work, int* d_info, cudaStream_t s,
                          long long polls) {
    // work: lu_work_bytes_f32(n, nb) bytes, 256-byte aligned: panel staging, then the
    // tensor-core split operands, then the cooperative panel's candidates and barrier
    void* split = reinterpret_cast<char*>(work) + split_offset(n, nb);
    void* coop = reinterpret_cast<char*>(work) + coop_offset(n, nb);
    return lu_factor<float>(A, n, piv, nb, work, d_info, split, coop, s, polls);
}
size_t lu_solve_work_bytes(int64_t n, size_t tsize) {
    return 2 * tsize * (size_t)n + 16 + 3 * sizeof(int) + 256;
}

size_t residual_work_bytes(int64_t n) {
    return sizeof(double) * (size_t)((n + kResChunk - 1) / kResChunk) * (size_t)n + 256;
}

cudaError_t lu_make_perm(const int32_t* piv, int64_t n, int32_t* perm, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const size_t bytes = sizeof(int32_t) * (size_t)n;
    if (bytes <= 200 * 1024) {
        // set for the current device on every call (an attribute is per device)
        NB_TRY(cudaFuncSetAttribute(k_make_perm_smem, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
        k_make_perm_smem<<<1, 1024, bytes, s>>>(piv, n, perm);
    } else {
        k_make_perm_global<<<1, 1, 0, s>>>(piv, n, perm);
    }
    return cudaGetLastError();
}

cudaError_t lu_solve_f64(const double* LU, int64_t n, const int32_t* perm, double* b, void* work, cudaStream_t s,
                         long long polls) {
    return lu_solve<double>(LU, n, perm, b, static_cast<double*>(work), s, polls);
}
cudaError_t lu_solve_f32(const float* LU, int64_t n, const int32_t* perm, float* b, void* work, cudaStream_t s,
                         long long polls) {
    return lu_solve<float>(LU, n, perm, b, static_cast<float*>(work), s, polls);
}
const int* lu_solve_err_flag(const void* work, int64_t n, size_t tsize) {
    // as laid out by lu_solve: y, z (n values each), then 16-byte aligned the two tickets and the error flag
    const uintptr_t fo = ((uintptr_t)static_cast<const char*>(work) + 2 * tsize * (size_t)n + 15) & ~(uintptr_t)15;
    return reinterpret_cast<const int*>(fo) + 2;
}
cudaError_t gemv_residual(const double* K, int64_t n, const double* x, const double* b, double* r, void* work,
                          cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const int64_t nchunk = (n + kResChunk - 1) / kResChunk;
    double* part = static_cast<double*>(work);
    dim3 grid((unsigned)((n + kResRows - 1) / kResRows), (unsigned)nchunk);
    k_residual_partial<<<grid, kResRows, 0, s>>>(K, n, x, part);
    k_residual_final<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(part, nchunk, n, b, r);
    return cudaGetLastError();
}
cudaError_t copy_f64_to_f32(const double* a, float* b, int64_t n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_f64_to_f32<<<(unsigned)std::min<int64_t>(65535, (n + 255) / 256), 256, 0, s>>>(a, b, n);
    return cudaGetLastError();
}
cudaError_t ir_update(double* x, const float* d, int64_t n, double* d_norms, cudaStream_t s) {
    NB_TRY(cudaMemsetAsync(d_norms, 0, 2 * sizeof(double), s));
    k_ir_update<<<(unsigned)std::min<int64_t>(1024, (n + 255) / 256), 256, 0, s>>>(x, d, n, d_norms);
    return cudaGetLastError();
}
cudaError_t vec_absmax(const double* a, int64_t n, double* out, cudaStream_t s) {
    NB_TRY(cudaMemsetAsync(out, 0, sizeof(double), s));
    k_absmax<<<(unsigned)std::min<int64_t>(1024, (n + 255) / 256), 256, 0, s>>>(a, n, out);
    return cudaGetLastError();
}

// ---- several right-hand sides (columns of leading dimension n), kMR per pass
size_t lu_solve_multi_work_bytes(int64_t n, size_t tsize) {
    return 2 * tsize * (size_t)n * kMR + 16 + 3 * sizeof(int) + 256;
}
static int* multi_tickets(const void* work, int64_t n, size_t tsize) {
    // y, z (n x kMR values each), then the 16-byte aligned tickets of both sweeps and the error flag
    const uintptr_t fo =
        ((uintptr_t)static_cast<const char*>(work) + 2 * tsize * (size_t)n * kMR + 15) & ~(uintptr_t)15;
    return reinterpret_cast<int*>(fo);
}
const int* lu_solve_multi_err_flag(const void* work, int64_t n, size_t tsize) {
    return multi_tickets(work, n, tsize) + 2;
}
template <typename T>
static cudaError_t lu_solve_multi(const T* LU, int64_t n, const int32_t* perm, T* B, int64_t nrhs, void* work,
                                  cudaStream_t s, long long polls) {
    if (n == 0 || nrhs == 0) return cudaSuccess;
    const int64_t nblk = (n + kTB - 1) / kTB;
    T* y = static_cast<T*>(work);
    T* z = y + n * kMR;
    int* tickets = multi_tickets(work, n, sizeof(T));
    int* err = tickets + 2;
    NB_TRY(cudaMemsetAsync(err, 0, sizeof(int), s));
    const long long limit = polls > 0 ? polls : kSvSpinLimit;
    // set for the current device on every call (an attribute is per device)
    const size_t smem = trsm_smem_bytes<T>();
    NB_TRY(cudaFuncSetAttribute(k_trsm<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    for (int64_t c0 = 0; c0 < nrhs; c0 += kMR) {
        const int nr = (int)std::min<int64_t>(kMR, nrhs - c0);
        T* b = B + c0 * n;
        NB_TRY(cudaMemsetAsync(tickets, 0, 2 * sizeof(int), s));
        k_permute_m<T><<<(unsigned)((n * nr + 255) / 256), 256, 0, s>>>(b, perm, n, nr, y, z);
        k_trsm<T><<<(unsigned)nblk, kSvThreads, smem, s>>>(LU, n, nblk, 1, y, z, b, nr, tickets, err, limit);
        k_trsm<T><<<(unsigned)nblk, kSvThreads, smem, s>>>(LU, n, nblk, 0, z, b, nullptr, nr, tickets + 1, err, limit);
        NB_TRY(cudaGetLastError());
    }
    return cudaSuccess;
}
cudaError_t lu_solve_multi_f64(const double* LU, int64_t n, const int32_t* perm, double* B, int64_t nrhs, void* work,
                               cudaStream_t s, long long polls) {
    return lu_solve_multi<double>(LU, n, perm, B, nrhs, work, s, polls);
}
cudaError_t lu_solve_multi_f32(const float* LU, int64_t n, const int32_t* perm, float* B, int64_t nrhs, void* work,
                               cudaStream_t s, long long polls) {
    return lu_solve_multi<float>(LU, n, perm, B, nrhs, work, s, polls);
}
size_t residual_multi_work_bytes(int64_t n) {
    return sizeof(double) * (size_t)((n + kResChunk - 1) / kResChunk) * kMR * (size_t)n + 256;
}
cudaError_t gemv_residual_multi(const double* K, int64_t n, const double* X, int64_t nrhs, const double* B, double* R,
                                void* work, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    const int64_t nchunk = (n + kResChunk - 1) / kResChunk;
    double* part = static_cast<double*>(work);
    for (int64_t c0 = 0; c0 < nrhs; c0 += kMR) {
        const int nr = (int)std::min<int64_t>(kMR, nrhs - c0);
        dim3 grid((unsigned)((n + kResRows - 1) / kResRows), (unsigned)nchunk);
        switch (nr) {  // the column count as a template argument: no predicated lanes
            case 1: launch_residual_partial_m<1>(grid, s, K, n, X + c0 * n, part); break;
            case 2: launch_residual_partial_m<2>(grid, s, K, n, X + c0 * n, part); break;
            case 3: launch_residual_partial_m<3>(grid, s, K, n, X + c0 * n, part); break;
            case 4: launch_residual_partial_m<4>(grid, s, K, n, X + c0 * n, part); break;
            case 5: launch_residual_partial_m<5>(grid, s, K, n, X + c0 * n, part); break;
            case 6: launch_residual_partial_m<6>(grid, s, K, n, X + c0 * n, part); break;
            case 7: launch_residual_partial_m<7>(grid, s, K, n, X + c0 * n, part); break;
            default: launch_residual_partial_m<8>(grid, s, K, n, X + c0 * n, part); break;
        }
        k_residual_final_m<<<(unsigned)((n * nr + 255) / 256), 256, 0, s>>>(part, nchunk, n, nr, B + c0 * n,
                                                                           R + c0 * n);
        NB_TRY(cudaGetLastError());
    }
    return cudaSuccess;
}
cudaError_t ir_update_multi(double* X, const float* D, int64_t n, int64_t nrhs, uint64_t active, double* d_norms,
                            cudaStream_t s) {
    if (nrhs > 64) return cudaErrorInvalidValue;
    NB_TRY(cudaMemsetAsync(d_norms, 0, 2 * sizeof(double) * (size_t)nrhs, s));
    if (n == 0) return cudaSuccess;
    for (int64_t c0 = 0; c0 < nrhs; c0 += kMR) {
        const int nr = (int)std::min<int64_t>(kMR, nrhs - c0);
        const uint32_t act = (uint32_t)((active >> c0) & ((1ull << nr) - 1ull));
        if (!act) continue;
        dim3 grid((unsigned)std::min<int64_t>(1024, (n + 255) / 256), (unsigned)nr);
        k_ir_update_m<<<grid, 256, 0, s>>>(X + c0 * n, D + c0 * n, n, act, d_norms + 2 * c0);
        NB_TRY(cudaGetLastError());
    }
    return cudaSuccess;
}

}  // namespace nb
