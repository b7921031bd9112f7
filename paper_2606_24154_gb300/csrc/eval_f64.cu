// eval_f64.cu -- FP64 evaluation and influence-matrix fill kernels.
//
// Evaluation (Eq. Potential / Eq. Field with element charge densities):
//   phi(x) = ke sum_j sigma_j sum_k Phi'(x - t_k; j),  E(x) likewise with E'.
// One thread per target (body f64_block in eval_blocks.cuh); element tiles are staged in
// shared memory (broadcast reads); the image sum of one element is accumulated in its
// local frame and rotated once.
//
// Fill (Eq. Matrix, collocation at centroids):
//   conductor row i:  K_ij = ke sum_k Phi'(c_i - t_k; j)
//   interface row i:  K_ij = ke sum_k n_i . E'(c_i - t_k; j) + delta_ij diag_i
// Thread per row i (coalesced column-major stores K[i + j n]), grid.y over column chunks.
#include "eval_blocks.cuh"

namespace nb {

namespace {

constexpr int kThreads = 128;
constexpr int kFillBlocks = 3;  // resident fill blocks per SM
constexpr int kF64Blocks = 3;  // resident evaluation blocks per SM (168 registers a thread)

// Block u takes unit u of `plan`: whole groups of points, then element pieces of the left-over
// groups (see split_plan).  1,500 points x 4,632 elements x 25 copies: 516 ms with a thread per
// point in 12 blocks, 42 ms in pieces.
__global__ void __launch_bounds__(kEvalThreads, kF64Blocks)
    k_eval_f64(const Elem* __restrict__ el, const double* __restrict__ sigma, int64_t n_el, const ImageTable img,
               const double* __restrict__ pts, int64_t npts, const SplitPlan plan, Sum4* __restrict__ part,
               double* __restrict__ phi, double* __restrict__ E) {
    const SplitUnit t = split_unit(plan, blockIdx.x, n_el);
    const int64_t p = t.group * kEvalThreads + threadIdx.x;
    {
        const bool active = p < npts;
        const double Px = active ? pts[3 * p] : 0.0, Py = active ? pts[3 * p + 1] : 0.0,
                     Pz = active ? pts[3 * p + 2] : 0.0;
        f64_sum(el, sigma, t.e0, t.e1, img, Px, Py, Pz);
    }
    if (p >= npts) return;
    if (t.whole)
        store_far(pts, phi, E, p, total_slot()->s);
    else
        part[(t.r * kEvalThreads + threadIdx.x) * plan.np + t.piece] = total_slot()->s;
}

// the left-over groups' points: their pieces added along the summation tree, a warp per point
__global__ void __launch_bounds__(256) k_f64_reduce(const double* __restrict__ pts, int64_t npts, const SplitPlan plan,
                                                    const Sum4* __restrict__ part, double* __restrict__ phi,
                                                    double* __restrict__ E) {
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t p = plan.Gm * kEvalThreads + w;
    if (p >= npts) return;
    const Sum4 tot = split_reduce(part + w * plan.np, plan.np, plan.leaf);
    if ((threadIdx.x & 31) == 0) store_far(pts, phi, E, p, tot);
}

// Bound by the FP64 pipe: 4,632 elements x 25 copies take 121 ms, 4.4e9 pairs a second, where
// the general form alone took 298 ms (114 FP64 instructions a pair, counted: 0.85 of the measured
// 0.619e12 a second).  Conductor rows form the potential only and interface rows the
// field only; the row's normal is rotated into the column's frame once per (row, column), so that
// an image of an interface row adds three products.
__global__ void __launch_bounds__(kThreads, kFillBlocks)
    k_fill_f64(const Elem* __restrict__ el, const double* __restrict__ diag_in, int64_t n, const ImageTable img, int cols,
               double* __restrict__ K) {
    __shared__ Tile64 s_t;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool active = i < n;
    double cx = 0.0, cy = 0.0, cz = 0.0, nx = 0.0, ny = 0.0, nz = 0.0, diag = 0.0;
    int bc = 0;
    if (active) {
        const Elem& ei = el[i];
        cx = ei.c[0];
        cy = ei.c[1];
        cz = ei.c[2];
        nx = ei.ey[0];
        ny = ei.ey[1];
        nz = ei.ey[2];
        bc = ei.bc;
        diag = diag_in[i];  // (eps_a + eps_b) / (2 eps0 (eps_b - eps_a)) on interface rows, else 0
    }
    const double ke = 1.0 / (4.0 * kPi * kEps0);
    const int64_t j0 = (int64_t)blockIdx.y * cols;
    const int64_t j1 = min(n, j0 + cols);
    for (int64_t base = j0; base < j1; base += kTile64) {
        const int cnt = (int)min((int64_t)kTile64, j1 - base);
        load_tile64(s_t, el, base, cnt, img);
        for (int jj = 0; jj < cnt; ++jj) {
            const Elem& e = s_t.el[jj];
            const int64_t j = base + jj;
            double X0, Y0, Z0;
            to_local(e, __dsub_rn(cx, e.o[0]), __dsub_rn(cy, e.o[1]), __dsub_rn(cz, e.o[2]), X0, Y0, Z0);
            double acc = 0.0, f, gx, gy, gz;
            if (bc == NEBEM_CONDUCTOR) {
                for (int k = 0; k < img.n; ++k) {
                    const double* tau = s_t.tau[jj][k];
                    const bool self = (i == j) && (k == img.k0);
                    elem_at_f64<true, false>(e, s_t.edge[jj], __dsub_rn(X0, tau[0]), self ? 0.0 : __dsub_rn(Y0, tau[1]),
                                             __dsub_rn(Z0, tau[2]), f, gx, gy, gz);
                    acc = __dadd_rn(acc, f);
                }
            } else {
                double mx, my, mz;
                to_local(e, nx, ny, nz, mx, my, mz);
                for (int k = 0; k < img.n; ++k) {
                    const double* tau = s_t.tau[jj][k];
                    const bool self = (i == j) && (k == img.k0);
                    elem_at_f64<false, true>(e, s_t.edge[jj], __dsub_rn(X0, tau[0]), self ? 0.0 : __dsub_rn(Y0, tau[1]),
                                             __dsub_rn(Z0, tau[2]), f, gx, gy, gz);
                    acc = __dadd_rn(acc, __fma_rn(mx, gx, __fma_rn(my, gy, __dmul_rn(mz, gz))));
                }
            }
            if (active) K[i + j * n] = (i == j) ? fma(ke, acc, diag) : ke * acc;
        }
    }
}

__global__ void k_element_influence(const Elem* __restrict__ el, int64_t n_el, const double* __restrict__ pts,
                                    int64_t npts, double* __restrict__ phi, double* __restrict__ E) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_el * npts) return;
    const int64_t e = t / npts, p = t % npts;
    const Elem& el_e = el[e];
    double f, gx, gy, gz;
    elem_local_f64(el_e, pts[3 * p], pts[3 * p + 1], pts[3 * p + 2], false, f, gx, gy, gz);
    phi[t] = f;
    E[3 * t] = fma(gx, el_e.ex[0], fma(gy, el_e.ey[0], gz * el_e.ez[0]));
    E[3 * t + 1] = fma(gx, el_e.ex[1], fma(gy, el_e.ey[1], gz * el_e.ez[1]));
    E[3 * t + 2] = fma(gx, el_e.ex[2], fma(gy, el_e.ey[2], gz * el_e.ez[2]));
}

}  // namespace

size_t f64_part_bytes(int64_t npts, int sms, int64_t n_el) {
    const SplitPlan plan = split_plan((npts + kEvalThreads - 1) / kEvalThreads, kF64Blocks * (int64_t)sms, n_el,
                                      (int64_t)(kPartMax / sizeof(Sum4)));
    return sizeof(Sum4) * (size_t)(plan.R * plan.np * kEvalThreads);
}

cudaError_t launch_eval_f64(const Elem* el, const double* sigma, int64_t n_el, const ImageTable& img,
                            const double* pts, int64_t npts, double* phi, double* E, int sms, void* part,
                            size_t part_bytes, cudaStream_t s) {
    if (npts == 0) return cudaSuccess;
    const int64_t gb = kF64Blocks * (int64_t)sms;
    const SplitPlan plan = split_plan((npts + kEvalThreads - 1) / kEvalThreads, gb, n_el,
                                      (int64_t)(part_bytes / sizeof(Sum4)));
    const int64_t units = plan.Gm + plan.R * plan.np;
    k_eval_f64<<<(unsigned)units, kEvalThreads, 0, s>>>(el, sigma, n_el, img, pts, npts, plan,
                                                        static_cast<Sum4*>(part), phi, E);
    if (plan.R > 0)
        k_f64_reduce<<<(unsigned)((plan.R * kEvalThreads + 7) / 8), 256, 0, s>>>(
            pts, npts, plan, static_cast<const Sum4*>(part), phi, E);
    return cudaGetLastError();
}

cudaError_t sm_count(int* sms) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    return e != cudaSuccess ? e : cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
}

cudaError_t fill_cols(int64_t n, int rows, int per_sm, int* cols) {
    int sms = 0;
    const cudaError_t e = sm_count(&sms);
    if (e != cudaSuccess) return e;
    *cols = 64;
    while (*cols > 2 && (n + rows - 1) / rows * ((n + *cols - 1) / *cols) < 2 * (int64_t)per_sm * sms) *cols /= 2;
    return cudaSuccess;
}

cudaError_t launch_fill_f64(const Elem* el, const double* diag, int64_t n, const ImageTable& img, double* K,
                            cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    int cols = 0;
    const cudaError_t e = fill_cols(n, kThreads, kFillBlocks, &cols);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((n + kThreads - 1) / kThreads), (unsigned)((n + cols - 1) / cols));
    k_fill_f64<<<grid, kThreads, 0, s>>>(el, diag, n, img, cols, K);
    return cudaGetLastError();
}

cudaError_t launch_element_influence(const Elem* el, int64_t n_el, const double* pts, int64_t npts,
                                     double* phi, double* E, cudaStream_t s) {
    const int64_t total = n_el * npts;
    if (total == 0) return cudaSuccess;
    k_element_influence<<<(unsigned)((total + 127) / 128), 128, 0, s>>>(el, n_el, pts, npts, phi, E);
    return cudaGetLastError();
}

}  // namespace nb
