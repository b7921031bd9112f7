// lu_tc64.cu -- trailing update of the FP64 LU on the 5th-generation tensor cores:
// C[M x N] -= A[M x K] B[K x N], K <= 64, column-major FP64, the update that follows each panel
// (Sec. 4.1 / Alg. 1; almost all of the 2/3 n^3 operations).
//
// The FP64 pipe does two multiply-adds per SM and clock (1.24 TFLOP/s on 152 SMs).  Here the
// product is formed exactly from integer digits on the FP16 tensor pipe, after the error-free
// splitting of Ozaki, Ogita, Oishi and Rump ("Error-free transformations of matrix multiplication
// by using fast routines of matrix multiplication", Numer. Algorithms 59, 2012):
//   - Scaling.  g_k = exponent of the largest |B_kj| of row k; A_ik 2^g_k is scaled per row and
//     B_kj 2^-g_k per column, both by powers of two, to 62-bit fixed point.  With g_k the split is
//     unchanged when rows or columns of the factored matrix are scaled (conductor rows and interface
//     rows differ by a factor of 1e6), which a split by rows and columns alone is not.
//   - Digits.  Eight balanced base-256 digits (-128 .. 127) per number, exact in FP16: 64 bits,
//     where an FP64 number has 53.
//   - Products.  The 36 digit products s + t <= 7 accumulate by d = s + t in eight FP32 accumulators:
//     |sum| <= 8 terms x 64 x 2^14 = 2^23, so every partial sum is an integer that FP32 holds exactly.
//     The products left out are below 2^-53 of (row scale x column scale) in the worst case and
//     about 2^-59 for digits of random sign.
//   - Epilogue.  The eight integers are joined to one 64-bit integer, rounded once to FP64 and
//     subtracted from C by one fma: two FP64 instructions per element instead of 64.
// Against 64 fmas in a row, whose roundings add up, the result is the more accurate one.
//
// One CTA per SM (192 KB of shared memory): the A digits of 128 rows (128 KB) once, then the
// B digits of 64 columns (64 KB) tile by tile; 144 MMAs (M 128, N 64, K 16) per tile into the whole of
// tensor memory (8 x 64 columns).  The next tile's B digits are copied while the epilogue runs.
// The epilogue's FP64 and conversion instructions and the MMAs' shared-memory reads take about
// the same time, and share a CTA in turn.  Every wait is bounded.
//
// Measured, LU of a random matrix of order 6145: the updates 142 ms on the FP64 pipe, 15 ms here; the
// whole factorisation 234 -> 40 ms, |P A - L U| / |A| 3.4e-14 -> 2.7e-14.
#include <cuda_fp16.h>

#include <algorithm>

#include "nb_internal.h"
#include "tcgen05.cuh"

namespace nb {

namespace {

constexpr int kDM = 128, kDN = 64, kDK = 64, kDig = 8;
constexpr int kDThreads = 256;
constexpr uint32_t kDLbo = 128;                       // next core matrix (8 rows x 8 halves) along K
constexpr uint32_t kDSbo = (kDK / 8) * 128;           // next 8-row group
constexpr uint32_t kDPlaneA = kDM * kDK * 2;          // 16 KB: one digit of the A tile
constexpr uint32_t kDPlaneB = kDN * kDK * 2;          // 8 KB
constexpr uint32_t kDTileA = kDig * kDPlaneA, kDTileB = kDig * kDPlaneB;
constexpr uint32_t kDSmem = kDTileA + kDTileB + 64;
constexpr int kNonFinite = 1 << 24;                   // exponent mark of a row or column with Inf or NaN

// instruction descriptor, kind::f16: D = F32 (bits 4-5 = 1), A = B = F16 (0), both K-major, N >> 3 at
// bits 17-22, M >> 4 at bits 24-28
constexpr uint32_t kDIdesc = (1u << 4) | ((uint32_t)(kDN >> 3) << 17) | ((uint32_t)(kDM >> 4) << 24);

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

// x 2^shift as a 62-bit fixed-point number: mantissa m (53 bits) shifted by sh = 9 - (top - e)
__device__ __forceinline__ long long fixed62(unsigned long long bits, int sh) {
    const unsigned long long mag = bits & ~(1ull << 63);
    unsigned long long m = mag & ((1ull << 52) - 1);
    if (mag >> 52) m |= 1ull << 52;
    if (sh >= 0)
        m <<= sh;
    else
        m = sh > -62 ? (m + (1ull << (-sh - 1))) >> -sh : 0;
    return (bits >> 63) ? -(long long)m : (long long)m;
}

// eight numbers (consecutive k) to eight digit planes, 16 bytes each
__device__ __forceinline__ void store_digits(const unsigned long long (&v)[8], const int (&sh)[8],
                                             unsigned char* __restrict__ dst, uint32_t plane) {
    long long x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = fixed62(v[q], sh[q]);
#pragma unroll
    for (int s = kDig - 1; s >= 0; --s) {
        alignas(16) __half h[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int d = s ? (int)(signed char)(x[q] & 255) : (int)x[q];
            x[q] = (x[q] - d) >> 8;
            h[q] = __int2half_rn(d);
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
    int sh[8], top = 0;
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
        for (int q = 0; q < 8; ++q) sh[q] = top >= kNonFinite ? -64 : 9 - (top - sh[q]);
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (!(v[q] << 1)) sh[q] = 0;
        const int r = (int)(row % kDM);
        store_digits(v, sh, da + (row / kDM) * (size_t)kDTileA + (r >> 3) * kDSbo + warp * kDLbo + (r & 7) * 16,
                     kDPlaneA);
    } else {
        const int64_t col = ((int64_t)blockIdx.x - blocks_a) * 32 + warp * 4 + lane / 8;
        const int kg = lane % 8;
        top = -8192;  // a zero column's mark: below every exponent
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
        for (int q = 0; q < 8; ++q) sh[q] = top >= kNonFinite ? -64 : 9 - (top - sh[q]);
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

// c - (sum of acc_d 256^(7-d)) 2^(56 + e0), the eight sums given as exact FP32 integers, e = the
// exponents of row and column added up.
__device__ __forceinline__ double take_off(double c, const uint32_t (&a)[kDig], int e) {
    int i[kDig];
#pragma unroll
    for (int d = 0; d < kDig; ++d) i[d] = __float2int_rn(__uint_as_float(a[d]));
    const long long H = (long long)((i[0] << 8) + i[1]) * 65536 + ((i[2] << 8) + i[3]);
    const long long L = (long long)((i[4] << 8) + i[5]) * 65536 + ((i[6] << 8) + i[7]);
    // |H| < 2^42.2 (top digits <= 65); the low part rounded to nearest: cut off, it would lean every
    // element of every update the same way (the residual of n = 6145 was 2.4 times the chain's)
    const double t = (double)((H << 20) + ((L + 2048) >> 12));  // units of 2^68 of the digit product
    const int x = e - 2100 + 1023;
    if (x > 0 && x < 2047) return __fma_rn(-t, __longlong_as_double((long long)x << 52), c);
    if (e >= kNonFinite / 2) return __longlong_as_double(0x7ff8000000000000ll);
    return c - scalbn(t, max(-3000, e - 2100));
}

// (bounds: 168 registers, so that a CTA of the next panel fits beside this one)
__global__ void __launch_bounds__(384, 1)
    k_tc_update_f64(int64_t M, int64_t N, const unsigned char* __restrict__ da, const unsigned char* __restrict__ db,
                    const int* __restrict__ ea, const int* __restrict__ eb, double* __restrict__ C, int64_t ldc,
                    int64_t tile0, int64_t tile1, int tpc, int* __restrict__ err) {
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
            for (int d = 0; d < kDig; ++d)
                for (int s = 0; s <= d; ++s)
                    for (int ks = 0; ks < kDK / 16; ++ks) {
                        const uint64_t ad = digit_desc(smem_u32(sA + s * kDPlaneA) + (uint32_t)ks * 2u * kDLbo);
                        const uint64_t bd = digit_desc(smem_u32(sB + (d - s) * kDPlaneB) + (uint32_t)ks * 2u * kDLbo);
                        asm volatile(
                            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(
                                tmem + (uint32_t)(d * kDN)),
                            "l"(ad), "l"(bd), "r"(kDIdesc), "r"((s | ks) ? 1u : 0u));
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
                if (row < M && n0 + cb + j < N)
                    C[row + (n0 + cb + j) * ldc] = take_off(c[cb + j], a, er + eb[n0 + cb + j]);
            }
        }
        // the next tile's MMAs overwrite the accumulators: every warp's reads come first
        asm volatile("tcgen05.fence::before_thread_sync;");
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

cudaError_t tc_apply_f64(int64_t M, int64_t N, int64_t c0, int64_t c1, double* C, int64_t ldc, void* work, int* err,
                         cudaStream_t s) {
    c1 = std::min(c1, N);
    if (M <= 0 || c0 >= c1) return cudaSuccess;
    if (c0 % kDN || !work) return cudaErrorInvalidValue;
    const Tables64 t = tables64(M, N, work);
    // set for the current device on every call (an attribute is per device)
    cudaError_t e = cudaFuncSetAttribute(k_tc_update_f64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDSmem);
    if (e != cudaSuccess) return e;
    // column tiles per CTA: about three CTAs per SM in all, at most 8 tiles each
    const int64_t tiles_m = pad_to(M, kDM) / kDM, tile0 = c0 / kDN, tile1 = (c1 + kDN - 1) / kDN, tiles_n = tile1 - tile0;
    const int64_t tpc = std::max<int64_t>(1, std::min<int64_t>(8, tiles_m * tiles_n / (3 * 152)));
    dim3 grid((unsigned)tiles_m, (unsigned)((tiles_n + tpc - 1) / tpc));
    k_tc_update_f64<<<grid, kDThreads, kDSmem, s>>>(M, N, t.da, t.db, t.ea, t.eb, C, ldc, tile0, tile1, (int)tpc, err);
    return cudaGetLastError();
}

}  // namespace nb
