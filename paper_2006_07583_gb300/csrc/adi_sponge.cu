// adi_sponge.cu -- absorbing layers: Cerjan's damping, the technique Sec. 2.1 names for the
// CFD formulation.  After every full step, each field value at a point whose distance to the
// nearest wall is delta cells, delta < width, is multiplied by g = exp(-(a (width - delta))^2);
// the pressure's wall values (the Dirichlet data) are left alone.
//
// The line kernels carry (a, v, w*) from step to step, and pointwise damping of the natural
// fields does not commute with the non-local derivatives inside a and w*.  So a simulation with
// layers writes its natural fields every step; this kernel damps them (u, w natural; v, which
// the x-line stage leaves in natural form, in place) and the prologue kernels then rebuild
// the carried state from them, exactly as adi_set_fields does (adi_api.cu).
#include <cuda_runtime.h>

#include "../../include/adi.h"
#include "adi_internal.h"

namespace adi {

namespace {

// Coordinate in cells of index k along an axis of n cells: nodes for CFD and for the unstaggered
// axis of an MFD velocity; cell centres plus the two walls for a staggered MFD axis.
__device__ __forceinline__ double cell_coord(int method, bool staggered, int k, int n) {
    if (method == ADI_CFD || !staggered) return (double)k;
    if (k == 0) return 0.0;
    if (k == n + 1) return (double)n;
    return (double)k - 0.5;
}

// The factor at distance d of one axis.  It rises with d, so the factor at the nearest wall's distance is
// the smaller of the two axes' factors.
__device__ __forceinline__ double damping(double x, int n, double width, double a) {
    const double d = fmin(x, (double)n - x);
    if (d >= width) return 1.0;
    const double q = a * (width - d);
    return exp(-q * q);
}

// The axes' factors in FP64: staggered x (ldu values), nodal x (ldv), staggered y (rows_u), nodal y (rows_w).
__global__ void sponge_axes_kernel(SpongeRec r, double *g) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < r.ldu) g[k] = damping(cell_coord(r.method, true, k, r.nx), r.nx, r.width, r.a);
    g += r.ldu;
    if (k < r.ldv) g[k] = damping(cell_coord(r.method, false, k, r.nx), r.nx, r.width, r.a);
    g += r.ldv;
    if (k < r.rows_u) g[k] = damping(cell_coord(r.method, true, k, r.ny), r.ny, r.width, r.a);
    g += r.rows_u;
    if (k < r.rows_w) g[k] = damping(cell_coord(r.method, false, k, r.ny), r.ny, r.width, r.a);
}

// blockIdx.z: 0 = u (natural, rows_u x ldu, interior only), 1 = v (rows_v x ldv, leading
// dimension ldvp), 2 = w (natural, rows_w x ldw).  A block takes 256 columns and kSpongeRows rows, with the axes'
// factors from the table built when the layers were set; points outside the layers cost two integer tests.  (An
// FP64 exponential and a 64-bit division per point took 37 us a step for 640 x 640 cells, exponentials per
// axis and block 13 us, this 6.8 us.)
constexpr int kSpongeRows = 8;
__device__ __forceinline__ bool is_one(double g) { return __double2hiint(g) == 0x3ff00000; }  // g <= 1
template <typename T>
__global__ void __launch_bounds__(256) sponge_kernel(SpongeRec r) {
    const int f = blockIdx.z;
    const int rows = f == 0 ? r.rows_u : (f == 1 ? r.rows_v : r.rows_w);
    const int cols = f == 0 ? r.ldu : (f == 1 ? r.ldv : r.ldw);
    const long long ld = f == 0 ? r.ldu : (f == 1 ? r.ldvp : r.ldw);
    T *x = (T *)(f == 0 ? r.uo : (f == 1 ? r.v : r.wo));
    // u: both axes staggered (MFD); v: x on nodes, y staggered; w: x staggered, y on nodes
    const double *tx = r.g + (f == 1 ? r.ldu : 0), *ty = r.g + r.ldu + r.ldv + (f == 2 ? r.rows_u : 0);
    const int i0 = blockIdx.y * kSpongeRows, j = blockIdx.x * 256 + threadIdx.x;
    if (j >= cols) return;
    const double gx = tx[j];
#pragma unroll
    for (int k = 0; k < kSpongeRows; ++k) {
        const int i = i0 + k;
        if (i >= rows) break;
        const double gy = ty[i];
        if (is_one(gx) && is_one(gy)) continue;
        if (f == 0 && (i == 0 || j == 0 || i == rows - 1 || j == cols - 1)) continue;  // walls
        const T val = (T)((double)x[(size_t)i * ld + j] * fmin(gx, gy));
        x[(size_t)i * ld + j] = val;
        // v's first and last rows are not lines of the x-line stage, which therefore never
        // carries them from one copy to the other: both copies take the damped value
        if (f == 1 && (i == 0 || i == rows - 1)) ((T *)r.v_other)[(size_t)i * ld + j] = val;
    }
}

}  // namespace

template <typename T>
cudaError_t launch_sponge(const SpongeRec &r, cudaStream_t s) {
    const int rows = r.rows_u > r.rows_w ? r.rows_u : r.rows_w, cols = r.ldu > r.ldv ? r.ldu : r.ldv;
    const dim3 grid((unsigned)((cols + 255) / 256), (unsigned)((rows + kSpongeRows - 1) / kSpongeRows), 3);
    sponge_kernel<T><<<grid, 256, 0, s>>>(r);
    return cudaGetLastError();
}

size_t sponge_axes_values(const SpongeRec &r) { return (size_t)r.ldu + r.ldv + r.rows_u + r.rows_w; }
cudaError_t launch_sponge_axes(const SpongeRec &r, double *g, cudaStream_t s) {
    const int x = r.ldu > r.ldv ? r.ldu : r.ldv, y = r.rows_u > r.rows_w ? r.rows_u : r.rows_w, n = x > y ? x : y;
    sponge_axes_kernel<<<(n + 127) / 128, 128, 0, s>>>(r, g);
    return cudaGetLastError();
}

template cudaError_t launch_sponge<float>(const SpongeRec &, cudaStream_t);
template cudaError_t launch_sponge<double>(const SpongeRec &, cudaStream_t);

}  // namespace adi
