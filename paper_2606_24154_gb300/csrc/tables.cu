// tables.cu -- per-geometry tables made on the device from the element records: the cell lists of
// the near-pair searches, and the two-float element records, Gauss nodes and image shifts of the
// mixed fill and of the refined evaluation.  On the host (and copied over, 28 MB) they were most of
// the 40 ms that a mixed solve of a 9,996-element cell with 25 copies spent outside its kernels; 7 ms
// are left.
#include "eval_blocks.cuh"
#include "geometry.h"

namespace nb {

namespace {

// ---------------------------------------------------------------- cell list
__device__ __forceinline__ int32_t cell_of(const Elem& e, const ImageTable& img, int k, const NearGrid& g) {
    int64_t cc[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double f = floor(__dmul_rn(__dsub_rn(__dadd_rn(e.c[a], img.t[k][a]), g.origin[a]), g.inv_h));
        cc[a] = (int64_t)fmin(fmax(f, 0.0), (double)g.dims[a] - 1.0);
    }
    return (int32_t)((cc[2] * g.dims[1] + cc[1]) * g.dims[0] + cc[0]);
}

// key of image i: its cell, then its index, so that the sorted list (and with it the order of every
// near sum) is the same on every run; the keys from `total` on fill up the sort's length
__global__ void k_cell_keys(const Elem* __restrict__ el, int64_t total, int64_t padded, const ImageTable img,
                            const NearGrid g, long long* __restrict__ keys, int32_t* __restrict__ count) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= padded) return;
    if (i >= total) {
        keys[i] = 0x7fffffffffffffffll;
        return;
    }
    const int64_t j = i / img.n;
    const int32_t c = cell_of(el[j], img, (int)(i - j * img.n), g);
    keys[i] = ((long long)c << 32) | i;
    atomicAdd(&count[c], 1);
}
__global__ void k_cell_items(const long long* __restrict__ keys, int64_t total, int32_t* __restrict__ items) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < total) items[i] = (int32_t)(keys[i] & 0xffffffffll);
}

// exclusive scan of n counts in place: sums of 1024, one block over the sums, then every block its own
__device__ __forceinline__ int32_t block_scan(int32_t v, int32_t& total) {  // 1024 threads: exclusive prefix
    __shared__ int32_t s_w[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) s_w[w] = inc;
    __syncthreads();
    if (w == 0) {
        int32_t x = s_w[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t u = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += u;
        }
        s_w[lane] = x;
    }
    __syncthreads();
    total = s_w[31];
    const int32_t before = w ? s_w[w - 1] : 0;
    __syncthreads();
    return before + inc - v;
}
__global__ void __launch_bounds__(1024) k_scan_sums(const int32_t* __restrict__ a, int64_t n, int32_t* __restrict__ sums) {
    const int64_t i = (int64_t)blockIdx.x * 1024 + threadIdx.x;
    int32_t t;
    block_scan(i < n ? a[i] : 0, t);
    if (threadIdx.x == 0) sums[blockIdx.x] = t;
}
__global__ void __launch_bounds__(1024) k_scan_one(int32_t* __restrict__ sums, int64_t n) {
    int32_t run = 0;
    for (int64_t b = 0; b < n; b += 1024) {
        const int64_t i = b + threadIdx.x;
        int32_t t;
        const int32_t x = block_scan(i < n ? sums[i] : 0, t);
        if (i < n) sums[i] = run + x;
        run += t;
    }
}
// start[i] = exclusive prefix, start[n] = the total
__global__ void __launch_bounds__(1024) k_scan_apply(int32_t* __restrict__ start, int64_t n,
                                                     const int32_t* __restrict__ sums) {
    const int64_t i = (int64_t)blockIdx.x * 1024 + threadIdx.x;
    const int32_t v = i < n ? start[i] : 0;
    int32_t t;
    const int32_t x = sums[blockIdx.x] + block_scan(v, t);
    if (i < n) {
        start[i] = x;
        if (i == n - 1) start[n] = x + v;
    }
}

// ---------------------------------------------------------------- fill tables
__device__ __forceinline__ float4 hi4(const double (&v)[3]) {
    return make_float4(__double2float_rn(v[0]), __double2float_rn(v[1]), __double2float_rn(v[2]), 0.f);
}
__device__ __forceinline__ float4 lo4(const double (&v)[3], const float4& h) {
    return make_float4(__double2float_rn(v[0] - (double)h.x), __double2float_rn(v[1] - (double)h.y),
                       __double2float_rn(v[2] - (double)h.z), 0.f);
}

__global__ void k_fill_records(const Elem* __restrict__ el, int64_t n, FillEl* __restrict__ fe) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const Elem& e = el[j];
    FillEl r;
    r.ch = hi4(e.c), r.cl = lo4(e.c, r.ch);
    r.ch.w = (float)e.rho;
    r.exh = hi4(e.ex), r.exl = lo4(e.ex, r.exh);
    r.eyh = hi4(e.ey), r.eyl = lo4(e.ey, r.eyh);
    r.ezh = hi4(e.ez), r.ezl = lo4(e.ez, r.ezh);
    const double ra = kFillRatioA * e.rho, rb = kFillRatioB * e.rho, rc = kFillRatioC * e.rho;
    r.hdr = make_float4((float)(ra * ra), (float)(rb * rb), (float)(rc * rc), e.nv == 4 ? 5.f : 3.f);
    fe[j] = r;
}

__global__ void k_fill_tau(const Elem* __restrict__ el, int64_t total, const ImageTable img, float4* __restrict__ tau) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int64_t j = i / img.n;
    const int k = (int)(i - j * img.n);
    double v[3];
    to_local(el[j], img.t[k][0], img.t[k][1], img.t[k][2], v[0], v[1], v[2]);
    const float4 h = hi4(v);
    tau[2 * i] = h;
    tau[2 * i + 1] = lo4(v, h);
}

// the node pairs of the three tiers, one thread per (element, pair)
constexpr int kPairsAll = kFillPairsA + kFillPairsB + kFillPairsC;
static_assert(kFillNodeRec == 4 * kPairsAll, "node record");

__global__ void k_fill_nodes(const Elem* __restrict__ el, int64_t n, const GaussRules g, float4* __restrict__ nodes) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * kPairsAll) return;
    const int64_t j = i / kPairsAll;
    const int p = (int)(i - j * kPairsAll);
    const Elem& e = el[j];
    const bool quad = e.nv == 4;
    const int tier = p < kFillPairsA ? 0 : p < kFillPairsA + kFillPairsB ? 1 : 2;
    const int q = p - (tier == 0 ? 0 : tier == 1 ? kFillPairsA : kFillPairsA + kFillPairsB);
    const int m = tier == 0 ? 3 : tier == 1 ? 4 : 6;  // tensor order (triangles: the 6-point rule in tier 0)
    const int cnt = tier == 0 && !quad ? 6 : m * m;
    float4* dst = nodes + j * kFillNodeRec + 4 * p;
    if (2 * q >= cnt) {
        for (int t = 0; t < 4; ++t) dst[t] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    const double* x = tier == 0 ? g.x3 : tier == 1 ? g.x4 : g.x6;
    const double* w = tier == 0 ? g.w3 : tier == 1 ? g.w4 : g.w6;
    const double dc[3] = {e.c[0] - e.o[0], e.c[1] - e.o[1], e.c[2] - e.o[2]};
    const double cx = dc[0] * e.ex[0] + dc[1] * e.ex[1] + dc[2] * e.ex[2];
    const double cz = dc[0] * e.ez[0] + dc[1] * e.ez[1] + dc[2] * e.ez[2];
    float h[2][4], l[2][4];
    for (int lane = 0; lane < 2; ++lane) {
        const bool pad = 2 * q + lane >= cnt;  // an odd count: the last node again, of weight 0
        const int node = pad ? 2 * q : 2 * q + lane;
        double px, pz, wt;
        if (quad) {
            // tensor Gauss-Legendre on the bilinear map q0 + s e1 + t e3 + s t tw, weight ws wt |x_s x x_t|
            const double e1x = e.qx[1] - e.qx[0], e1z = e.qz[1] - e.qz[0];
            const double e3x = e.qx[3] - e.qx[0], e3z = e.qz[3] - e.qz[0];
            const double twx = e.qx[2] - e.qx[1] - e3x, twz = e.qz[2] - e.qz[1] - e3z;
            const double s = x[node / m], t = x[node % m];
            px = e.qx[0] + s * e1x + t * e3x + s * t * twx;
            pz = e.qz[0] + s * e1z + t * e3z + s * t * twz;
            const double sx = e1x + t * twx, sz = e1z + t * twz, tx = e3x + s * twx, tz = e3z + s * twz;
            wt = w[node / m] * w[node % m] * fabs(sx * tz - sz * tx);
        } else {
            const double area = 0.5 * e.twoA[0];
            if (tier == 0) {
                double bc[3] = {g.tri_a[node / 3], g.tri_a[node / 3], g.tri_a[node / 3]};
                bc[node % 3] = 1.0 - 2.0 * g.tri_a[node / 3];
                px = bc[0] * e.qx[0] + bc[1] * e.qx[1] + bc[2] * e.qx[2];
                pz = bc[0] * e.qz[0] + bc[1] * e.qz[1] + bc[2] * e.qz[2];
                wt = g.tri_w[node / 3] * area;
            } else {
                // collapsed (Duffy) product rule: q0 + s e1 + t (1 - s) e2, weight 2 ws wt (1 - s) A
                const double s = x[node / m], t = x[node % m] * (1.0 - s);
                px = e.qx[0] + s * (e.qx[1] - e.qx[0]) + t * (e.qx[2] - e.qx[0]);
                pz = e.qz[0] + s * (e.qz[1] - e.qz[0]) + t * (e.qz[2] - e.qz[0]);
                wt = 2.0 * w[node / m] * w[node % m] * (1.0 - s) * area;
            }
        }
        const double sx = cx - px, sz = cz - pz;
        const double v[4] = {2.0 * sx, 2.0 * sz, sx * sx + sz * sz, pad ? 0.0 : wt};
        for (int c = 0; c < 4; ++c) {
            h[lane][c] = __double2float_rn(v[c]);
            l[lane][c] = __double2float_rn(v[c] - (double)h[lane][c]);
        }
    }
    dst[0] = make_float4(h[0][0], h[1][0], h[0][1], h[1][1]);
    dst[1] = make_float4(h[0][2], h[1][2], h[0][3], h[1][3]);
    dst[2] = make_float4(l[0][0], l[1][0], l[0][1], l[1][1]);
    dst[3] = make_float4(l[0][2], l[1][2], l[0][3], l[1][3]);
}

unsigned blocks_of(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

size_t cell_list_work_bytes(int64_t total, int64_t ncell) {
    return sizeof(long long) * (size_t)vox_pad_len(total) + sizeof(int32_t) * (size_t)((ncell + 1023) / 1024);
}

cudaError_t launch_cell_list(const Elem* el, int64_t n, const ImageTable& img, const NearGrid& grid,
                             int32_t* cell_start, int32_t* cell_items, void* work, cudaStream_t s) {
    const int64_t total = n * img.n, ncell = (int64_t)grid.dims[0] * grid.dims[1] * grid.dims[2];
    cudaError_t e = cudaMemsetAsync(cell_start, 0, sizeof(int32_t) * (size_t)(ncell + 1), s);
    if (e != cudaSuccess || total == 0) return e;
    const int64_t P = vox_pad_len(total);
    long long* keys = static_cast<long long*>(work);
    int32_t* sums = reinterpret_cast<int32_t*>(keys + P);
    const unsigned sb = blocks_of(ncell, 1024);
    k_cell_keys<<<blocks_of(P, 256), 256, 0, s>>>(el, total, P, img, grid, keys, cell_start);
    k_scan_sums<<<sb, 1024, 0, s>>>(cell_start, ncell, sums);
    k_scan_one<<<1, 1024, 0, s>>>(sums, sb);
    k_scan_apply<<<sb, 1024, 0, s>>>(cell_start, ncell, sums);
    e = launch_sort_keys(keys, P, s);
    if (e != cudaSuccess) return e;
    k_cell_items<<<blocks_of(total, 256), 256, 0, s>>>(keys, total, cell_items);
    return cudaGetLastError();
}

cudaError_t launch_fill_tables(const Elem* el, int64_t n, const ImageTable& img, FillEl* fe, float4* nodes,
                               float4* tau, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_fill_records<<<blocks_of(n, 128), 128, 0, s>>>(el, n, fe);
    k_fill_tau<<<blocks_of(n * img.n, 256), 256, 0, s>>>(el, n * img.n, img, tau);
    k_fill_nodes<<<blocks_of(n * kPairsAll, 256), 256, 0, s>>>(el, n, gauss_rules(), nodes);
    return cudaGetLastError();
}

}  // namespace nb
