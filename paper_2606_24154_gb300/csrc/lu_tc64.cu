// lu_tc64.cu -- trailing update of the FP64 LU on the 5th-generation tensor cores:
// C[M x N] -= A[M x K] B[K x N], K <= 64, column-major FP64, the update that follows each panel
// (Sec. 4.1 / Alg. 1; almost all of the 2/3 n^3 operations).
//
// The FP64 pipe does two multiply-adds per SM and clock (1.24 TFLOP/s on 152 SMs).  Here most elements of
// the product are formed from integer digits on the BF16 tensor pipe, after the splitting of Ozaki, Ogita,
// Oishi and Rump ("Error-free transformations of matrix multiplication by using fast routines of matrix
// multiplication", Numer. Algorithms 59, 2012), and the others by a chain of FP64 fmas:
//   - Scaling.  g_k = exponent of the largest |B_kj| of row k; A_ik 2^g_k is scaled per row and
//     B_kj 2^-g_k per column, both by powers of two, to 63-bit fixed point.  With g_k the split is unchanged
//     when rows of the factored matrix are scaled, or dense columns (conductor rows and interface rows
//     differ by a factor of 1e6).
//   - Digits.  Eight balanced base-256 digits (-128 .. 128) per number, digit s held as digit x 256^-s, exact
//     in BF16: 64 bits, where an FP64 number has 53.  An entry more than 10 binary places below the largest
//     of its (scaled) row or column loses its last bits: at most 2^-64 of the scale.
//   - Products.  The 36 digit products s + t <= 7 accumulate by d = s + t in eight FP32 accumulators:
//     |sum| <= 8 terms x 64 x 2^14 = 2^23 units, so every partial sum is an integer that FP32 holds exactly.
//     The seven of s + t = 8 (below 2^15 of the units of d = 7) go to the accumulator of d = 7 first, where
//     they are kept to a unit at worst.  The 21 products left out are below 2^-63 of
//     row scale x column scale.
//   - Epilogue.  The eight sums are joined to one integer, cut to 62 bits, rounded once to FP64 and
//     subtracted from C by one fma: two FP64 instructions per element instead of 64.
//   - Elements that are small beside their row and column.  All errors above stay within 2^-57 of row scale x
//     column scale (64 terms with two entries off by 2^-64 each).  The chain's bound is 64 x 2^-53 of
//     |C_ij| + sum_k |A_ik B_kj|.  So where |C_ij| or the result's own sum reaches 2^-10 of row scale x column
//     scale, the digits keep the chain's bound element by element (their largest error there is a sixth of the
//     chain's).  The other elements (take_off: false), those of rows or columns that are not finite and those
//     at the ends of the exponent range are formed by fmas.  Random matrices: 5 in 100,000 elements; THGEM
//     cells of 4,632, 2,100 and 828 elements: 0.04, 0.13 and 0.7 %; two groups of rows and columns coupled by
//     1e-4 or less: the coupled half, which then costs what it costs on the FP64 pipe.
//
// One CTA per SM (192 KB of shared memory): the A digits of 128 rows (128 KB) once, then the
// B digits of 64 columns (64 KB) tile by tile; 172 MMAs (M 128, N 64, K 16) per tile into the whole of
// tensor memory (8 x 64 columns).  The next tile's B digits are copied while the epilogue runs.
// The epilogue's FP64 and conversion instructions and the MMAs' shared-memory reads take about
// the same time, and share a CTA in turn.  Every wait is bounded.
//
// Measured, LU of a random matrix of order 6145: 234 ms with the updates (142 ms) on the FP64 pipe, 41.4 ms so;
// with every second row and column in a group coupled by 1e-4 or 1e-12, 234 and 210 ms; one in 32, 234 and 73 ms.
#include <cuda_bf16.h>

#include <algorithm>

#include "nb_internal.h"
#include "tcgen05.cuh"

namespace nb {

namespace {

constexpr int kDM = 128, kDN = 64, kDK = 64, kDig = 8;
constexpr int kDThreads = 256;
constexpr uint32_t kDLbo = 128;                       // next core matrix (8 rows x 8 values) along K
constexpr uint32_t kDSbo = (kDK / 8) * 128;           // next 8-row group
constexpr uint32_t kDPlaneA = kDM * kDK * 2;          // 16 KB: one digit of the A tile
constexpr uint32_t kDPlaneB = kDN * kDK * 2;          // 8 KB
constexpr uint32_t kDTileA = kDig * kDPlaneA, kDTileB = kDig * kDPlaneB;
constexpr uint32_t kDSmem = kDTileA + kDTileB + 64;
constexpr int kNonFinite = 1 << 24;                   // exponent mark of a row or column with Inf or NaN
constexpr int kZeroMark = -16384;                     // of a row or column of zeros: below every exponent
constexpr int kFixed = 10;                            // binary places that the largest mantissa (53 bits) is raised by

// instruction descriptor, kind::f16: D = F32 (bits 4-5 = 1), A = B = BF16 (1 at bits 7-9 and 10-12), both
// K-major, N >> 3 at bits 17-22, M >> 4 at bits 24-28
constexpr uint32_t kDIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kDN >> 3) << 17) | ((uint32_t)(kDM >> 4) << 24);

__device__ __forceinline__ uint64_t digit_desc(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(kDLbo >> 4) << 16) | ((uint64_t)(kDSbo >> 4) << 32) |
           (1ull << 46);
}

// biased exponent, at least 1 (subnormal numbers and zero), of the magnitude's bits
__device__ __forceinline__ int bexp(unsigned long long mag) { return max(1, (int)(mag >> 52)); }

// g[k] = largest exponent of the finite entries of row k of B (g zeroed before)
__global__ void __launch_bounds__(256) k_row_exps(const double* __restrict__ B, int64_t ldb, int K, int64_t N,
                                                  int* __restrict__ g) {
    const int k = threadIdx.x % kDK;
    int e = 1;
    if (k < K)
        for (int64_t j = (int64_t)blockIdx.x * 4 + threadIdx.x / kDK; j < N; j += (int64_t)gridDim.x * 4) {
            const int b = bexp((unsigned long long)__double_as_longlong(B[k + j * ldb]) & ~(1ull << 63));
            if (b < 0x7ff) e = max(e, b);
        }
    if (k < K) atomicMax(&g[k], e);
}

// x 2^shift as a 63-bit fixed-point number: mantissa m (53 bits) shifted by sh = kFixed - (top - e)
__device__ __forceinline__ long long fixed63(unsigned long long bits, int sh) {
    const unsigned long long mag = bits & ~(1ull << 63);
    unsigned long long m = mag & ((1ull << 52) - 1);
    if (mag >> 52) m |= 1ull << 52;
    if (sh >= 0)
        m <<= sh;
    else
        m = sh > -62 ? (m + (1ull << (-sh - 1))) >> -sh : 0;
    return (bits >> 63) ? -(long long)m : (long long)m;
}

// 256^d, d <= 8
__host__ __device__ constexpr float pow256(int d) {
    float p = 1.f;
    for (int i = 0; i < d; ++i) p *= 256.f;
    return p;
}

// eight numbers (consecutive k) to eight digit planes (digit s x 256^-s), 16 bytes each
__device__ __forceinline__ void store_digits(const unsigned long long (&v)[8], const int (&sh)[8],
                                             unsigned char* __restrict__ dst, uint32_t plane) {
    long long x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = fixed63(v[q], sh[q]);
#pragma unroll
    for (int s = kDig - 1; s >= 0; --s) {
        alignas(16) __nv_bfloat16 h[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int d = s ? (int)(signed char)(x[q] & 255) : (int)x[q];
            x[q] = (x[q] - d) >> 8;
            h[q] = __float2bfloat16_rn((float)d * (1.f / pow256(s)));
        }
        *reinterpret_cast<uint4*>(dst + (size_t)s * plane) = *reinterpret_cast<const uint4*>(h);
    }
}

// The digit tiles of A (blocks [0, blocks_a), 32 rows each) and B (32 columns each), and the
// exponents ea[row], eb[column].  A: warp = eight consecutive k, lane = row.  B: eight lanes
// share a column, each eight consecutive k.
__global__ void __launch_bounds__(256) k_split_digits(const double* __restrict__ A, int64_t lda,
                                                      const double* __restrict__ B, int64_t ldb, int64_t M, int64_t N,
                                                      int K, const int* __restrict__ g, int64_t blocks_a,
                                                      unsigned char* __restrict__ da, unsigned char* __restrict__ db,
                                                      int* __restrict__ ea, int* __restrict__ eb) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long v[8];
    int sh[8], top = kZeroMark;
    if ((int64_t)blockIdx.x < blocks_a) {
        __shared__ int s_top[8][32];
        const int64_t row = (int64_t)blockIdx.x * 32 + lane;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int k = 8 * warp + q;
            v[q] = (row < M && k < K) ? (unsigned long long)__double_as_longlong(A[row + (int64_t)k * lda]) : 0ull;
            const unsigned long long mag = v[q] & ~(1ull << 63);
            sh[q] = bexp(mag) + (k < K ? g[k] : 1);
            if (mag >> 52 == 0x7ff)
                top = kNonFinite;
            else if (mag)
                top = max(top, sh[q]);
        }
        s_top[warp][lane] = top;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < 8; ++w) top = max(top, s_top[w][lane]);
        if (warp == 0) ea[row] = top;
#pragma unroll
        for (int q = 0; q < 8; ++q) sh[q] = top >= kNonFinite ? -64 : kFixed - (top - sh[q]);
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (!(v[q] << 1)) sh[q] = 0;
        const int r = (int)(row % kDM);
        store_digits(v, sh, da + (row / kDM) * (size_t)kDTileA + (r >> 3) * kDSbo + warp * kDLbo + (r & 7) * 16,
                     kDPlaneA);
    } else {
        const int64_t col = ((int64_t)blockIdx.x - blocks_a) * 32 + warp * 4 + lane / 8;
        const int kg = lane % 8;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int k = 8 * kg + q;
            v[q] = (col < N && k < K) ? (unsigned long long)__double_as_longlong(B[k + col * ldb]) : 0ull;
            const unsigned long long mag = v[q] & ~(1ull << 63);
            sh[q] = bexp(mag) - (k < K ? g[k] : 1);
            if (mag >> 52 == 0x7ff)
                top = kNonFinite;
            else if (mag)
                top = max(top, sh[q]);
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
        if (kg == 0) eb[col] = top;
#pragma unroll
        for (int q = 0; q < 8; ++q) sh[q] = top >= kNonFinite ? -64 : kFixed - (top - sh[q]);
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (!(v[q] << 1)) sh[q] = 0;
        const int c = (int)(col % kDN);
        store_digits(v, sh, db + (col / kDN) * (size_t)kDTileB + (c >> 3) * kDSbo + kg * kDLbo + (c & 7) * 16,
                     kDPlaneB);
    }
}

// v = columns [col, col + 8) of the warp's 32 lanes of tensor memory
__device__ __forceinline__ void tmem_ld8(uint32_t addr, uint32_t (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(addr));
}

// c -= T 2^(e - 2114), T = sum of acc_d 256^(7 - d) for the eight sums (integers; the last one with a
// fraction) of e = the exponents of row and column added up, row scale x column scale = 2^(e - 2044).
// false, and c as it was, where neither c nor the product reaches 2^-10 of the scale, or a power of two needed
// here is outside the normal range (also: a row or column that is not finite).
__device__ __forceinline__ bool take_off(double& c, const uint32_t (&a)[kDig], int e) {
    int i[kDig];
#pragma unroll
    for (int d = 0; d < kDig; ++d) i[d] = __float2int_rn(__uint_as_float(a[d]) * pow256(d));
    // T = 2^32 H + L, |H| < 2^44.1, |L| < 2^46.5
    const long long H = (long long)((i[0] << 8) + i[1]) * 65536 + ((i[2] << 8) + i[3]);
    const long long L = (long long)((i[4] << 8) + i[5]) * 65536 + ((i[6] << 8) + i[7]);
    const long long mag = H < 0 ? -H : H;
    const int ec = (__double2hiint(c) >> 20) & 0x7ff;
    if (e <= 1091 || e >= 3122 || (mag < (1ll << 28) && ec < e - 1031)) return false;
    // t = T 2^-s of at most 62 bits, rounded to nearest (cut off, it would lean every element of every
    // update the same way); |t| >= 2^60 where s > 0
    const int s = max(0, 35 - __clzll(mag));
    const long long t = (H << (32 - s)) + ((L + ((1ll << s) >> 1)) >> s);
    c = __fma_rn(-(double)t, __longlong_as_double((long long)(e - 2114 + 1023 + s) << 52), c);
    return true;
}

// The elements of the warp's 32 rows (from row0) and 32 columns (from n0) whose bits are set in the lanes'
// masks: C_ij -= sum_k A_ik B_kj by fmas.  Few rows of a column: the 64 terms of one element side by side
// (seven FP64 instructions); from kRedoRows on a chain per row (64 for all of them).
constexpr int kRedoRows = 9;
__device__ __noinline__ void redo(unsigned mask, int64_t row0, int64_t n0, int K, const double* __restrict__ A,
                                  int64_t lda, const double* __restrict__ B, int64_t ldb, double* C, int64_t ldc) {
    const int lane = threadIdx.x & 31;
    for (unsigned any = __reduce_or_sync(0xffffffffu, mask); any; any &= any - 1) {
        const int j = __ffs(any) - 1;
        const double* b = B + (n0 + j) * ldb;
        double* c = C + row0 + (n0 + j) * ldc;
        unsigned who = __ballot_sync(0xffffffffu, (mask >> j) & 1u);
        if (__popc(who) >= kRedoRows) {
            if ((who >> lane) & 1u) {
                double acc = 0.0;
#pragma unroll 8
                for (int k = 0; k < K; ++k) acc = __fma_rn(A[row0 + lane + (int64_t)k * lda], b[k], acc);
                c[lane] = __dsub_rn(c[lane], acc);
            }
            continue;
        }
        const double b0 = lane < K ? b[lane] : 0.0, b1 = lane + 32 < K ? b[lane + 32] : 0.0;
        for (; who; who &= who - 1) {
            const int r = __ffs(who) - 1;
            double v = lane < K ? __dmul_rn(A[row0 + r + (int64_t)lane * lda], b0) : 0.0;
            if (lane + 32 < K) v = __fma_rn(A[row0 + r + (int64_t)(lane + 32) * lda], b1, v);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
            if (lane == r) c[lane] = __dsub_rn(c[lane], v);
        }
    }
}

// (launched with kDThreads; bounds of 384 threads: 168 registers, so that a CTA of the next panel fits beside)
__global__ void __launch_bounds__(384, 1)
    k_tc_update_f64(int64_t M, int64_t N, int K, const double* __restrict__ A, int64_t lda,
                    const double* __restrict__ B, int64_t ldb, const unsigned char* __restrict__ da,
                    const unsigned char* __restrict__ db, const int* __restrict__ ea, const int* __restrict__ eb,
                    double* __restrict__ C, int64_t ldc, int64_t tile0, int64_t tile1, int tpc,
                    int* __restrict__ err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char* sA = smem;
    unsigned char* sB = smem + kDTileA;
    uint64_t* barA = reinterpret_cast<uint64_t*>(smem + kDTileA + kDTileB);
    uint64_t* barB = barA + 1;
    uint64_t* barM = barA + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(barA + 3);

    const int64_t t0 = tile0 + (int64_t)blockIdx.y * tpc;  // column tiles [tile0, tile1)
    const int nt = (int)min((int64_t)tpc, tile1 - t0);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto load_b = [&](int t) {
        mbar_expect(barB, kDTileB);
        bulk_load(sB, db + (size_t)(t0 + t) * kDTileB, kDTileB, barB);
    };
    if (tid == 0) {
        for (int b = 0; b < 3; ++b) mbar_init(barA + b);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_expect(barA, kDTileA);
        for (int q = 0; q < 2; ++q)
            bulk_load(sA + q * (kDTileA / 2), da + (size_t)blockIdx.x * kDTileA + q * (kDTileA / 2), kDTileA / 2, barA);
        load_b(0);
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kDig * kDN));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tmem_slot;

    const int64_t row = (int64_t)blockIdx.x * kDM + (warp & 3) * 32 + lane;
    const int half = (warp >> 2) * (kDN / 2);  // warps 4-7: the tile's second 32 columns
    const int er = ea[row];                    // the exponent tables are padded to whole tiles
    int ok = 1, loads = 1, commits = 0, used_b = 0, used_m = 0;
    for (int t = 0; t < nt && ok; ++t) {
        int w = mbar_wait(barB, (uint32_t)(t & 1));
        if (t == 0) w = w && mbar_wait(barA, 0);
        if (!__syncthreads_and(w)) {
            ok = 0;
            break;
        }
        ++used_b;
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (tid == 0) {
            bool first = true;
            for (int d = kDig; d >= 0; --d) {  // d = 8 before d = 7, into the same sums
                if (d < kDig - 1) first = true;
                for (int s = max(0, d - kDig + 1); s <= min(d, kDig - 1); ++s)
                    for (int ks = 0; ks < kDK / 16; ++ks) {
                        const uint64_t ad = digit_desc(smem_u32(sA + s * kDPlaneA) + (uint32_t)ks * 2u * kDLbo);
                        const uint64_t bd = digit_desc(smem_u32(sB + (d - s) * kDPlaneB) + (uint32_t)ks * 2u * kDLbo);
                        asm volatile(
                            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(
                                tmem + (uint32_t)(min(d, kDig - 1) * kDN)),
                            "l"(ad), "l"(bd), "r"(kDIdesc), "r"(first ? 0u : 1u));
                        first = false;
                    }
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                smem_u32(barM)));
        }
        ++commits;
        // C and the column exponents in flight while the tensor core works
        const int64_t n0 = (t0 + t) * kDN + half;
        double c[kDN / 2];
#pragma unroll
        for (int j = 0; j < kDN / 2; ++j) c[j] = (row < M && n0 + j < N) ? C[row + (n0 + j) * ldc] : 0.0;
        w = mbar_wait(barM, (uint32_t)(t & 1));
        if (!__syncthreads_and(w)) {
            ok = 0;
            break;
        }
        ++used_m;
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (t + 1 < nt) {
            if (tid == 0) load_b(t + 1);  // the MMAs have read B
            ++loads;
        }
        unsigned again = 0;  // columns of this thread's row that the digits are too coarse for
#pragma unroll
        for (int cb = 0; cb < kDN / 2; cb += 8) {
            uint32_t v[kDig][8];
#pragma unroll
            for (int d = 0; d < kDig; ++d)
                tmem_ld8(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(d * kDN + half + cb), v[d]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int d = 0; d < kDig; ++d)  // the values exist from here on
#pragma unroll
                for (int j = 0; j < 8; ++j) asm volatile("" : "+r"(v[d][j]));
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                uint32_t a[kDig];
#pragma unroll
                for (int d = 0; d < kDig; ++d) a[d] = v[d][j];
                const int e = er + eb[n0 + cb + j];  // (padded to whole tiles)
                if (row < M && n0 + cb + j < N && e > kZeroMark / 2) {
                    if (take_off(c[cb + j], a, e))
                        C[row + (n0 + cb + j) * ldc] = c[cb + j];
                    else
                        again |= 1u << (cb + j);
                }
            }
        }
        // the next tile's MMAs overwrite the accumulators: every warp's reads come first
        asm volatile("tcgen05.fence::before_thread_sync;");
        if (__any_sync(0xffffffffu, again)) redo(again, row - lane, n0, K, A, lda, B, ldb, C, ldc);
    }
    if (!ok) {
        if (tid == 0) {
            atomicExch(err, 1);
            // what this CTA started ends (bounded) before its memory goes
            mbar_wait(barA, 0);
            if (loads > used_b) mbar_wait(barB, (uint32_t)(used_b & 1));
            if (commits > used_m) mbar_wait(barM, (uint32_t)(used_m & 1));
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kDig * kDN));
}

int64_t pad_to(int64_t n, int64_t q) { return (n + q - 1) / q * q; }

}  // namespace

size_t tc64_work_bytes(int64_t M, int64_t N) {
    const int64_t m = pad_to(M, kDM), n = pad_to(N, kDN);
    return (size_t)(m / kDM) * kDTileA + (size_t)(n / kDN) * kDTileB + sizeof(int) * (size_t)(m + n + kDK) + 256;
}

namespace {
struct Tables64 {
    unsigned char *da, *db;
    int *ea, *eb, *g;
};
Tables64 tables64(int64_t M, int64_t N, void* work) {
    const int64_t m = pad_to(M, kDM), n = pad_to(N, kDN);
    Tables64 t;
    t.da = static_cast<unsigned char*>(work);
    t.db = t.da + (size_t)(m / kDM) * kDTileA;
    t.ea = reinterpret_cast<int*>(t.db + (size_t)(n / kDN) * kDTileB);
    t.eb = t.ea + m;
    t.g = t.eb + n;
    return t;
}
}  // namespace

cudaError_t tc_split_f64(int64_t M, int64_t N, int64_t K, const double* A, int64_t lda, const double* B, int64_t ldb,
                         void* work, cudaStream_t s) {
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    if (K > kDK || !work) return cudaErrorInvalidValue;
    const int64_t m = pad_to(M, kDM), n = pad_to(N, kDN);
    const Tables64 t = tables64(M, N, work);
    cudaError_t e = cudaMemsetAsync(t.g, 0, sizeof(int) * kDK, s);
    if (e != cudaSuccess) return e;
    k_row_exps<<<(unsigned)std::min<int64_t>((N + 15) / 16, 304), 256, 0, s>>>(B, ldb, (int)K, N, t.g);
    k_split_digits<<<(unsigned)(m / 32 + n / 32), 256, 0, s>>>(A, lda, B, ldb, M, N, (int)K, t.g, m / 32, t.da, t.db,
                                                               t.ea, t.eb);
    return cudaGetLastError();
}

cudaError_t tc_apply_f64(int64_t M, int64_t N, int64_t K, int64_t c0, int64_t c1, const double* A, int64_t lda,
                         const double* B, int64_t ldb, double* C, int64_t ldc, void* work, int* err, cudaStream_t s) {
    c1 = std::min(c1, N);
    if (M <= 0 || c0 >= c1) return cudaSuccess;
    if (c0 % kDN || !work) return cudaErrorInvalidValue;
    const Tables64 t = tables64(M, N, work);
    // set for the current device on every call (an attribute is per device)
    int sms = 0;
    cudaError_t e = sm_count(&sms);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_tc_update_f64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDSmem);
    if (e != cudaSuccess) return e;
    // column tiles per CTA: about three CTAs per SM in all, at most 8 tiles each
    const int64_t tiles_m = pad_to(M, kDM) / kDM, tile0 = c0 / kDN, tile1 = (c1 + kDN - 1) / kDN, tiles_n = tile1 - tile0;
    const int64_t tpc = std::max<int64_t>(1, std::min<int64_t>(8, tiles_m * tiles_n / (3 * sms)));
    dim3 grid((unsigned)tiles_m, (unsigned)((tiles_n + tpc - 1) / tpc));
    k_tc_update_f64<<<grid, kDThreads, kDSmem, s>>>(M, N, (int)K, A, lda, B, ldb, t.da, t.db, t.ea, t.eb, C, ldc, tile0,
                                                    tile1, (int)tpc, err);
    return cudaGetLastError();
}

}  // namespace nb
