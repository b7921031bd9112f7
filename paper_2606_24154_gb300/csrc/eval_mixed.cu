// eval_mixed.cu -- mixed-precision evaluation kernels (bodies in eval_blocks.cuh): spatial
// binning of the targets, the FP32 far-field kernel over all (element, image) pairs, the
// FP64 near-pair kernel over the cell list, and the per-geometry two-float image-centroid
// table.
#include "eval_blocks.cuh"

namespace nb {

namespace {

constexpr int kFarBlocks = 6;  // resident far blocks per SM (80 registers a thread)

// Far part of every point: block u takes unit u of `plan` (whole groups, then pieces of the
// left-over groups).  Bound by the FP32 pipe where every SM has its six
// blocks; a thread's own chain of pairs takes as long on an idle SM as on a full one, so few
// points are spread over element pieces (see split_plan): 257 points of the 9,996-element
// cell x 25 copies took 71.2 ms in 3 blocks and take 0.63 ms in 939; 20,000 points 69 and 15 ms,
// 200,000 points 162 and 122 ms, 1e6 points 644 and 592 ms (with binning and near pairs).
__global__ void __launch_bounds__(kEvalThreads, kFarBlocks)
    k_eval_far(const GeomView g, const double* __restrict__ pts, const int32_t* __restrict__ order, int64_t npts,
               const SplitPlan plan, SumB* __restrict__ part, double* __restrict__ phi, double* __restrict__ E,
               float4* __restrict__ bound) {
    const int64_t n_el = g.n_el;
    const SplitUnit t = split_unit(plan, blockIdx.x, n_el);
    const int64_t i = t.group * kEvalThreads + threadIdx.x;
    {
        const bool active = i < npts;
        float phx, phy, phz, plx, ply, plz;
        load_point_2f(pts, active ? (int64_t)order[i] : 0, active, phx, phy, phz, plx, ply, plz);
        far_sum(g, phx, phy, phz, plx, ply, plz, t.e0, t.e1);
    }
    if (i >= npts) return;
    if (t.whole) {
        const int64_t p = order[i];
        store_far(pts, phi, E, p, total_slot()->s);
        store_bound(bound, p, total_slot()->b);
    } else {
        part[(t.r * kEvalThreads + threadIdx.x) * plan.np + t.piece] = *total_slot();
    }
}

// The same for few points: a unit is kFL points of one leaf (at most 32 elements), and a thread takes
// (point, element) pairs, two points of its element at a time, so that a launch does not end with
// threads that walk a whole leaf.  The chains over the elements follow from shared memory, a lane per
// quantity, with far_range's operations in its order (FP32 groups of kGroup elements within its tiles,
// the scales in FP32): the same bits.  Shared memory per tile of te elements in odd strides of float4, since
// the lanes read different elements.  10,000 elements x 25 copies: 5 points 0.33 ms by k_eval_far and
// 0.03 ms here, 64 points 0.49 and 0.13, 257 points 0.66 and 0.42.  The lanes of a warp take different tiers more
// often than neighbouring points do, so a point costs twice as much, and calls that share the GPU with
// others lose where k_eval_far's groups are full (257 points in several streams: 0.91 and 0.93 ms for the
// whole refined call): kFarLaneRounds units per resident block of k_eval_far, about 70 points.
constexpr int kFL = 8;                       // points of a unit
constexpr int kFLCentres = 1792;             // float4 of image centroids
constexpr int64_t kFarLaneRounds = 3;
__global__ void __launch_bounds__(kEvalThreads, 4)
    k_eval_far_lanes(const GeomView g, const double* __restrict__ pts, const int32_t* __restrict__ order, int64_t npts,
                     int64_t np, int te, SumB* __restrict__ part) {
    constexpr int kWarps = kEvalThreads / 32, kWP = kFL / kWarps, kF = 2 * kPairs0, kA = 2 * kPairsA;
    __shared__ float4 s_f[32][kF + 1], s_a[32][kA + 1], s_hdr[32], s_c[kFLCentres];
    __shared__ float2 s_sig[32];
    __shared__ int s_na[32];
    __shared__ float s_val[kWarps][kWP][32][7];  // sigma hi, lo, Phi', E'
    __shared__ float s_g[kFL][8];           // chains: the group's four sums, the four scales
    __shared__ double s_sum[kFL][4];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nimg = g.nimg, st = 2 * nimg + 1;
    const int64_t groups = (npts + kFL - 1) / kFL;
    const int64_t piece = blockIdx.x / groups, i0 = (blockIdx.x - piece * groups) * kFL;
    const int64_t e0 = piece * kLeafEl, e1 = min(e0 + (int64_t)kLeafEl, g.n_el);
    for (int c = lane; c < 8 * kWP; c += 32) s_g[w * kWP][c] = 0.f;
    for (int c = lane; c < 4 * kWP; c += 32) s_sum[w * kWP][c] = 0.0;
    __syncwarp();
    for (int64_t base = e0; base < e1; base += te) {
        const int cnt = (int)min((int64_t)te, e1 - base);
        __syncthreads();
        for (int i = threadIdx.x; i < cnt * kA; i += kEvalThreads) s_a[i / kA][i % kA] = g.far[base + i / kA].a[i % kA];
        for (int i = threadIdx.x; i < cnt * kF; i += kEvalThreads) s_f[i / kF][i % kF] = g.far[base + i / kF].f[i % kF];
        for (int i = threadIdx.x; i < cnt; i += kEvalThreads) {
            s_hdr[i] = g.far[base + i].hdr;
            s_na[i] = g.far[base + i].n_a;
            const double sd = fma(g.sigma[base + i], (double)g.far[base + i].wcorr, g.sigma[base + i]);
            const float sh = __double2float_rn(sd);
            s_sig[i] = make_float2(sh, __double2float_rn(sd - (double)sh));
        }
        for (int i = threadIdx.x; i < 2 * cnt * nimg; i += kEvalThreads)
            s_c[i / (2 * nimg) * st + i % (2 * nimg)] = g.cjk[2 * base * nimg + i];
        __syncthreads();
        // te = 32: a thread takes its element with the warp's two points; else 32 / te >= kWP points side by side
        static_assert(kWP == 2, "points of a warp");
        const int jj = lane % te;
        bool valid[kWP];
        float ph[kWP][6];
#pragma unroll
        for (int u = 0; u < kWP; ++u) {
            const int q = te == 32 ? u : lane / te;
            const int64_t i = i0 + w * kWP + q;
            valid[u] = jj < cnt && q < kWP && i < npts && (te == 32 || u == 0);
            load_point_2f(pts, valid[u] ? (int64_t)order[i] : 0, valid[u], ph[u][0], ph[u][1], ph[u][2], ph[u][3],
                          ph[u][4], ph[u][5]);
        }
        if (valid[0]) {
            const float4 hdr = s_hdr[jj];
            const bool rect = s_na[jj] == kPairsA;
            const FarNodes* fj = g.far + base + jj;
            const float4* cj = s_c + jj * st;
            float4 f0[kF];
#pragma unroll
            for (int i = 0; i < kF; ++i) f0[i] = s_f[jj][i];
            float2 lphi[kWP], lx[kWP], ly[kWP], lz[kWP];
#pragma unroll
            for (int u = 0; u < kWP; ++u) lphi[u] = lx[u] = ly[u] = lz[u] = make_float2(0.f, 0.f);
            for (int k = 0; k < nimg; ++k) {
                const float4 ch = cj[2 * k], cl = cj[2 * k + 1];
#pragma unroll
                for (int u = 0; u < kWP; ++u) {
                    if (!valid[u]) continue;
                    float dx, dy, dz;
                    const float d2 =
                        pair_d2(ph[u][0], ph[u][1], ph[u][2], ph[u][3], ph[u][4], ph[u][5], ch, cl, dx, dy, dz);
                    const float2 DX = make_float2(dx, dx), DY = make_float2(dy, dy), DZ = make_float2(dz, dz);
                    if (d2 >= hdr.x) {
                        pairs0_reg(f0, DX, DY, DZ, lphi[u], lx[u], ly[u], lz[u]);
                    } else if (d2 >= hdr.y) {
                        if (rect)
                            node_pairs<kPairsA>(s_a[jj], DX, DY, DZ, lphi[u], lx[u], ly[u], lz[u]);
                        else
                            node_pairs<3>(s_a[jj], DX, DY, DZ, lphi[u], lx[u], ly[u], lz[u]);
                    } else if (d2 >= hdr.z) {
                        node_pairs<kPairsB>(fj->b, DX, DY, DZ, lphi[u], lx[u], ly[u], lz[u]);
                    } else if (d2 >= hdr.w) {
                        node_pairs<kPairsC>(fj->c, DX, DY, DZ, lphi[u], lx[u], ly[u], lz[u]);
                    }
                    // nearer pairs: k_eval_near
                }
            }
            const float2 sg = s_sig[jj];
#pragma unroll
            for (int u = 0; u < kWP; ++u) {
                float* o = s_val[w][u][lane];
                o[0] = sg.x, o[1] = sg.y;
                o[2] = lphi[u].x + lphi[u].y, o[3] = lx[u].x + lx[u].y;
                o[4] = ly[u].x + ly[u].y, o[5] = lz[u].x + lz[u].y;
            }
        }
        __syncwarp();
        // chain c of a point: 0-3 phi and E, 4-7 the scales
        for (int l = lane; l < 8 * kWP; l += 32) {
            const int q = l / 8, c = l % 8, pt = w * kWP + q;
            const float(*r)[7] = te == 32 ? s_val[w][q] : s_val[w][0] + q * te;
            float x = s_g[pt][c];
            double sum = c < 4 ? s_sum[pt][c] : 0.0;
            for (int e = 0; e < cnt; ++e) {
                const float s = r[e][0];
                if (c < 4) {
                    const float f = r[e][2 + c];
                    x = fmaf(s, f, fmaf(r[e][1], f, x));
                    const int in_tile = ((int)(base - e0) + e) & (g.tile_el - 1);  // a power of two
                    if (in_tile % kGroup == kGroup - 1 || in_tile == g.tile_el - 1 || base + e == e1 - 1) {
                        sum += (double)x;
                        x = 0.f;
                    }
                } else {
                    const float a = c & 1 ? fabsf(r[e][3]) + fabsf(r[e][4]) + fabsf(r[e][5]) : fabsf(r[e][2]);
                    const float b = fabsf(s) * a;
                    if (c < 6) {
                        x += b;
                    } else {
                        const float v = b * kScaleSq;
                        x = fmaf(v, v, x);
                    }
                }
            }
            s_g[pt][c] = x;
            if (c < 4) s_sum[pt][c] = sum;
        }
        __syncwarp();
    }
    for (int l = lane; l < 8 * kWP; l += 32) {
        const int pt = w * kWP + l / 8, c = l % 8;
        const int64_t i = i0 + pt;
        if (i >= npts) continue;
        SumB* o = part + i * np + piece;
        if (c < 4)
            reinterpret_cast<double*>(&o->s)[c] = s_sum[pt][c];
        else
            reinterpret_cast<float*>(&o->b)[c - 4] = s_g[pt][c];
    }
}

// the left-over groups' points: their pieces added along the summation tree, a warp per point
__global__ void __launch_bounds__(256) k_far_reduce(const double* __restrict__ pts, const int32_t* __restrict__ order,
                                                    int64_t npts, const SplitPlan plan,
                                                    const SumB* __restrict__ part, double* __restrict__ phi,
                                                    double* __restrict__ E, float4* __restrict__ bound) {
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t i = plan.Gm * kEvalThreads + w;
    if (i >= npts) return;
    const SumB tot = split_reduce(part + w * plan.np, plan.np, plan.leaf);
    if ((threadIdx.x & 31) != 0) return;
    const int64_t p = order[i];
    store_far(pts, phi, E, p, tot.s);
    store_bound(bound, p, tot.b);
}

__global__ void __launch_bounds__(kEvalThreads) k_eval_near(const GeomView g, const ImageTable img,
                                                          const double* __restrict__ pts,
                                                          const int32_t* __restrict__ order, int64_t npts,
                                                          double* __restrict__ phi, double* __restrict__ E) {
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= npts) return;
    near_point(g, img, pts, (int64_t)order[w], phi, E);
}

// ---- spatial binning of the targets: counting sort by the Morton index of a 64^3 grid
// over the near-pair grid's box (points outside are clamped to the border cells).  Warps
// then hold nearby points, whose (element, image) pairs mostly fall in the same distance
// tier, so the tier branches stay converged.  The order only changes which lane evaluates
// a point, never the point's arithmetic; positions within a cell come from atomics and
// may differ between runs without changing any result.
constexpr int kBinBits = 6;
constexpr int kBins = 1 << (3 * kBinBits);

__device__ __forceinline__ uint32_t spread3(uint32_t v) {  // 6 bits -> every third bit
    uint32_t r = 0;
#pragma unroll
    for (int b = 0; b < kBinBits; ++b) r |= ((v >> b) & 1u) << (3 * b);
    return r;
}

__global__ void k_bin_keys(const double* __restrict__ pts, int64_t n, const NearGrid grid,
                           int32_t* __restrict__ key, int32_t* __restrict__ count) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t c[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double span = (double)grid.dims[a] / grid.inv_h;
        double f = floor((pts[3 * i + a] - grid.origin[a]) / span * (double)(1 << kBinBits));
        f = fmin(fmax(f, 0.0), (double)((1 << kBinBits) - 1));
        c[a] = (uint32_t)f;
    }
    const int32_t k = (int32_t)(spread3(c[0]) | (spread3(c[1]) << 1) | (spread3(c[2]) << 2));
    key[i] = k;
    atomicAdd(&count[k], 1);
}

// Exclusive scan of the kBins counts in two launches of kBins / 1024 blocks: every block's
// sum of its 1024 counts, then every block scans its own counts from the sum of the blocks before
// it.  (One block for all 262,144 counts took 0.30 ms, in a chain of dependent loads.)
constexpr int kScanBlocks = kBins / 1024;
static_assert(kScanBlocks <= 1024, "one thread per block sum");

__device__ __forceinline__ int32_t warp_sum(int32_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__global__ void __launch_bounds__(256) k_bin_sums(const int32_t* __restrict__ count, int32_t* __restrict__ sums) {
    __shared__ int32_t s_w[8];
    const int4 c = reinterpret_cast<const int4*>(count)[blockIdx.x * 256 + threadIdx.x];
    const int32_t v = warp_sum(c.x + c.y + c.z + c.w);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t t = 0;
        for (int k = 0; k < 8; ++k) t += s_w[k];
        sums[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(1024) k_bin_scan(int32_t* __restrict__ count, const int32_t* __restrict__ sums) {
    __shared__ int32_t s_w[32], s_b[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int32_t before = ((int)threadIdx.x < kScanBlocks && threadIdx.x < blockIdx.x) ? sums[threadIdx.x] : 0;
    const int32_t bs = warp_sum(before);
    const int64_t i = (int64_t)blockIdx.x * 1024 + threadIdx.x;
    const int32_t c = count[i];
    int32_t inc = c;  // inclusive scan of the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) s_w[w] = inc;
    if (lane == 0) s_b[w] = bs;
    __syncthreads();
    const int32_t base = warp_sum(s_b[lane]) + warp_sum(lane < w ? s_w[lane] : 0);
    count[i] = base + inc - c;
}

__global__ void k_bin_scatter(const int32_t* __restrict__ key, int64_t n, int32_t* __restrict__ next,
                              int32_t* __restrict__ order) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    order[atomicAdd(&next[key[i]], 1)] = (int32_t)i;
}

// Two-float image centroids, entry (j, k) at 2 * (j * nimg + k): hi then lo.
__global__ void k_image_centroids(const Elem* __restrict__ el, int64_t n, const ImageTable img,
                                  float4* __restrict__ cjk) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * img.n) return;
    const int64_t j = i / img.n;
    const int k = (int)(i - j * img.n);
    float h[3], l[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) split2f(el[j].c[a] + img.t[k][a], h[a], l[a]);
    cjk[2 * i] = make_float4(h[0], h[1], h[2], 0.f);
    cjk[2 * i + 1] = make_float4(l[0], l[1], l[2], 0.f);
}

// Distance-tier code of every (point, element, image) pair, as the evaluation decides it:
// 0 tier 0, 1 tier a, 2 tier b, 3 tier c, 4 FP64 near pair.
__global__ void k_pair_tiers(const FarNodes* __restrict__ far, const float4* __restrict__ cjk, int64_t n_el, int nimg,
                             const double* __restrict__ pts, int64_t npts, uint8_t* __restrict__ codes) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= npts * n_el * nimg) return;
    const int64_t p = t / (n_el * nimg);
    const int64_t jk = t - p * (n_el * nimg);
    const int64_t j = jk / nimg;
    float phx, phy, phz, plx, ply, plz;
    split2f(pts[3 * p], phx, plx);
    split2f(pts[3 * p + 1], phy, ply);
    split2f(pts[3 * p + 2], phz, plz);
    float dx, dy, dz;
    const float d2 = pair_d2(phx, phy, phz, plx, ply, plz, cjk[2 * jk], cjk[2 * jk + 1], dx, dy, dz);
    const float4 h = far[j].hdr;
    codes[t] = (d2 >= h.x) ? 0 : (d2 >= h.y) ? 1 : (d2 >= h.z) ? 2 : (d2 >= h.w) ? 3 : 4;
}

}  // namespace

cudaError_t launch_pair_tiers(const FarNodes* far, const float4* cjk, int64_t n_el, int nimg, const double* pts,
                              int64_t npts, uint8_t* codes, cudaStream_t s) {
    const int64_t total = npts * n_el * nimg;
    if (total == 0) return cudaSuccess;
    k_pair_tiers<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(far, cjk, n_el, nimg, pts, npts, codes);
    return cudaGetLastError();
}

cudaError_t launch_image_centroids(const Elem* el, int64_t n, const ImageTable& img, float4* cjk, cudaStream_t s) {
    const int64_t total = n * img.n;
    if (total == 0) return cudaSuccess;
    k_image_centroids<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(el, n, img, cjk);
    return cudaGetLastError();
}

GeomView make_view(const Elem* el, const FarNodes* far, const float4* cjk, const double* sigma, int64_t n_el,
                   const ImageTable& img, const NearGrid& grid, const int32_t* cell_start, const int32_t* cell_items) {
    GeomView g;
    g.el = el;
    g.far = far;
    g.cjk = cjk;
    g.sigma = sigma;
    g.cell_start = cell_start;
    g.cell_items = cell_items;
    g.n_el = n_el;
    g.nimg = img.n;
    // largest power of two <= min(kTileMax, kCjkMax / images): divides the chunk width
    int t = 1;
    while (t * 2 <= kTileMax && t * 2 <= kCjkMax / img.n) t *= 2;
    g.tile_el = t;
    g.grid = grid;
    return g;
}

static size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

MixedScratch mixed_scratch(void* base, int64_t npts) {
    char* p = static_cast<char*>(base);
    MixedScratch m;
    const size_t n = (size_t)npts;
    m.count = reinterpret_cast<int32_t*>(p);
    p += align256(sizeof(int32_t) * kBins);
    m.key = reinterpret_cast<int32_t*>(p);
    p += align256(sizeof(int32_t) * n);
    m.order = reinterpret_cast<int32_t*>(p);
    p += align256(sizeof(int32_t) * n);
    m.bound = reinterpret_cast<float4*>(p);
    p += align256(sizeof(float4) * n);
    m.list = reinterpret_cast<int32_t*>(p);
    p += align256(sizeof(int32_t) * n);
    m.list2 = reinterpret_cast<int32_t*>(p);
    p += align256(sizeof(int32_t) * n);
    m.list_p = reinterpret_cast<int32_t*>(p);
    p += align256(sizeof(int32_t) * n);
    m.list_e = reinterpret_cast<int32_t*>(p);
    p += align256(sizeof(int32_t) * n);
    m.n_list = reinterpret_cast<int32_t*>(p);
    p += 256;
    m.bin_sums = reinterpret_cast<int32_t*>(p);
    return m;
}

size_t eval_mixed_scratch_bytes(int64_t npts) {
    const size_t n = (size_t)npts;
    return align256(sizeof(int32_t) * kBins) + 6 * align256(sizeof(int32_t) * n) + align256(sizeof(float4) * n) +
           256 + align256(sizeof(int32_t) * kScanBlocks);
}

size_t far_part_bytes(int64_t npts, int sms, int64_t n_el) {
    return split_part_bytes<SumB>(npts, kFarBlocks * (int64_t)sms, n_el);
}

cudaError_t launch_eval_mixed(const Elem* el, const FarNodes* far, const float4* cjk, const double* sigma,
                              int64_t n_el, const ImageTable& img, const NearGrid& grid, const int32_t* cell_start,
                              const int32_t* cell_items, const double* pts, int64_t npts, double* phi, double* E,
                              const MixedScratch& ms, int sms, void* part, size_t part_bytes, cudaStream_t s) {
    if (npts == 0) return cudaSuccess;
    if (npts > (int64_t)INT32_MAX) return cudaErrorInvalidValue;
    const GeomView g = make_view(el, far, cjk, sigma, n_el, img, grid, cell_start, cell_items);
    const unsigned pblocks = (unsigned)((npts + 255) / 256);
    cudaError_t e = cudaMemsetAsync(ms.count, 0, sizeof(int32_t) * kBins, s);
    if (e != cudaSuccess) return e;
    k_bin_keys<<<pblocks, 256, 0, s>>>(pts, npts, grid, ms.key, ms.count);
    k_bin_sums<<<kScanBlocks, 256, 0, s>>>(ms.count, ms.bin_sums);
    k_bin_scan<<<kScanBlocks, 1024, 0, s>>>(ms.count, ms.bin_sums);
    k_bin_scatter<<<pblocks, 256, 0, s>>>(ms.key, npts, ms.count, ms.order);
    const int64_t gb = kFarBlocks * (int64_t)sms;
    const SplitPlan plan = split_plan((npts + kEvalThreads - 1) / kEvalThreads, gb, n_el,
                                      (int64_t)(part_bytes / sizeof(SumB)));
    const int64_t units = plan.Gm + plan.R * plan.np;
    const int64_t lane_units = (npts + kFL - 1) / kFL * plan.np;
    if (plan.leaf && plan.Gm == 0 && lane_units < kFarLaneRounds * gb) {
        int te = 32;
        while (te > 1 && te * (2 * img.n + 1) > kFLCentres) te /= 2;
        k_eval_far_lanes<<<(unsigned)lane_units, kEvalThreads, 0, s>>>(g, pts, ms.order, npts, plan.np, te,
                                                                       static_cast<SumB*>(part));
    } else {
        k_eval_far<<<(unsigned)units, kEvalThreads, 0, s>>>(g, pts, ms.order, npts, plan, static_cast<SumB*>(part), phi,
                                                            E, ms.bound);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (plan.R > 0)
        k_far_reduce<<<(unsigned)((plan.R * kEvalThreads + 7) / 8), 256, 0, s>>>(
            pts, ms.order, npts, plan, static_cast<const SumB*>(part), phi, E, ms.bound);
    const int64_t near_blocks = (npts + kEvalThreads / 32 - 1) / (kEvalThreads / 32);
    k_eval_near<<<(unsigned)near_blocks, kEvalThreads, 0, s>>>(g, img, pts, ms.order, npts, phi, E);
    return cudaGetLastError();
}

}  // namespace nb
