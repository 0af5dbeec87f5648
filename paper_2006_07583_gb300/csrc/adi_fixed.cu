// adi_fixed.cu -- the paper's own way of solving the stage systems, for comparison with the
// exact line solves of the default path: the fixed-point iteration of Eq. 9 (Algorithms 3 and
// 4).  Each Peaceman-Rachford stage assembles its explicit right-hand side, then sweeps
//     u_{k+1} = a - alpha (Dv v_k),      v_{k+1} = v^m - beta (Du u_{k+1})
// along every line of its direction until the sum of the Frobenius norms of the two updates
// is at most eps, or kmax sweeps have run.  Dv, Du are the App. A compact operators
// (Pbar^{-1} Qbar, P^{-1} Q: a tridiagonal solve per application) or the App. B mimetic
// stencils (D4, G4).  The norm test runs on the device: every sweep's kernel reads a status
// word and returns at once when an earlier sweep has converged, so no host round trip sits
// between sweeps.  Natural (u, v, w) fields in row-major device arrays; one launch per sweep.
//
// A block takes up to four lines.  The stencils and updates are spread over its threads; the Thomas
// recurrences, which are serial along a line and are done in the order of a plain elimination, run on one thread per
// line out of shared memory, sixteen rows' operands loaded ahead; they bound it.  With everything on one thread per
// line in global memory (the paper's own decomposition) each row waited for memory several times: 1093 us a sweep for
// 512 lines of 512 cells, now 36 us.
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "../../include/adi.h"
#include "adi_internal.h"
#include "adi_line.cuh"
#include "adi_ops.cuh"

namespace adi {
namespace {

// Thomas factors of a tridiagonal operator of n rows: multipliers m_r (r >= 1), inverse
// pivots, super-diagonal.  Built on the host in FP64 from the App. A rows.
template <typename T>
struct FpTri {
    const T *m, *id, *c;
    int lo, hi;  // the rows lo .. hi-1 have the factors of row lo (the elimination settles within some 30 rows)
};

// Device-side convergence state of one stage's iteration.
struct FpState {
    double sum[2];  // squared Frobenius norms of the two updates of the current sweep
    unsigned arrived;  // blocks of the current sweep that have added theirs
    int k;          // sweeps done in this stage (its parity picks the current iterate's buffers)
    int done;       // the stage's iteration has stopped
    long long sweeps;  // sweeps over the whole call
};

// Lines of one direction: line l (first .. first + n - 1) of the pressure-like arrays starts
// at l * lsp with element stride esp, of the velocity arrays at l * lsv with stride esv.
struct FpLines {
    int first, n, N, L;  // L: last pressure index (N for CFD, N+1 for MFD)
    long long lsp, esp, lsv, esv;
};

__device__ __forceinline__ float mulr(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mulr(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fmar(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmar(double a, double b, double c) { return __fma_rn(a, b, c); }

// A block's share: `lines` (1, 2 or 4) lines from line0 on, nl of them in use; threads run along a line in whole
// warps where its elements are contiguous (unit), else with the lines side by side.
constexpr int kFpThreads = 256, kFpLines = 4;
struct FpShare {
    int lines, nl;
    long long line0;
    __device__ FpShare(const FpLines &g, int lines_) : lines(lines_) {
        const int at = blockIdx.x * lines;
        nl = min(lines, g.n - at);
        line0 = (long long)g.first + at;
    }
    __device__ int line(bool unit) const { return (unit ? threadIdx.x >> 5 : threadIdx.x) & (lines - 1); }
    __device__ int first(bool unit) const { return unit ? (threadIdx.x >> 5) / lines * 32 + (threadIdx.x & 31) : threadIdx.x / lines; }
    __device__ int step() const { return kFpThreads / lines; }
};

// Thomas solve in place, one thread per line: x[r], r < n, factors f (row r at index r).  The middle rows, whose
// factors are all the same, go in batches, the next batch's values loaded before this one's recurrence.
template <typename T>
__device__ void fp_thomas(T *x, int n, FpTri<T> f) {
    constexpr int U = 16;
    T v[U], w[U];
    T d = x[0];
    int r = 1;
    for (; r < f.lo; ++r) { d = fmar(-f.m[r], d, x[r]); x[r] = d; }
    if (r + U <= f.hi) {
        const T m = -f.m[r];
#pragma unroll
        for (int i = 0; i < U; ++i) v[i] = x[r + i];
        for (; r + U <= f.hi; r += U) {
            const bool more = r + 2 * U <= f.hi;
            if (more)
#pragma unroll
                for (int i = 0; i < U; ++i) w[i] = x[r + U + i];
#pragma unroll
            for (int i = 0; i < U; ++i) { d = fmar(m, d, v[i]); x[r + i] = d; }
            if (more)
#pragma unroll
                for (int i = 0; i < U; ++i) v[i] = w[i];
        }
    }
    for (; r < n; ++r) { d = fmar(-f.m[r], d, x[r]); x[r] = d; }
    d = mulr(d, f.id[n - 1]);
    x[n - 1] = d;
    for (r = n - 2; r >= f.hi; --r) { d = mulr(fmar(-f.c[r], d, x[r]), f.id[r]); x[r] = d; }
    if (r - U + 1 >= f.lo) {
        const T c = -f.c[r], id = f.id[r];
#pragma unroll
        for (int i = 0; i < U; ++i) v[i] = x[r - i];
        for (; r - U + 1 >= f.lo; r -= U) {
            const bool more = r - 2 * U + 1 >= f.lo;
            if (more)
#pragma unroll
                for (int i = 0; i < U; ++i) w[i] = x[r - U - i];
#pragma unroll
            for (int i = 0; i < U; ++i) { d = mulr(fmar(c, d, v[i]), id); x[r - i] = d; }
            if (more)
#pragma unroll
                for (int i = 0; i < U; ++i) v[i] = w[i];
        }
    }
    for (; r >= 0; --r) { d = mulr(fmar(-f.c[r], d, x[r]), f.id[r]); x[r] = d; }
}

// Du of the share's pressure lines u (global): CFD P^{-1} Q / h on nodes 0..N; MFD G4 / h.  Into x[l * pitch + j].
template <typename T>
__device__ void fp_du(int method, int N, T ih, const T *u, long long ls, long long es, const FpShare &sh, T *x, int pitch,
                      FpTri<T> P) {
    const int l = sh.line(es == 1);
    const T *ul = u + (sh.line0 + l) * ls;
    for (int j = sh.first(es == 1); j <= N && l < sh.nl; j += sh.step()) {
        T acc = T(0);
        if (method == kCFD && j > 0 && j < N) {
            acc = fmar(T(3), ul[(j + 1) * es], mulr(T(-3), ul[(j - 1) * es]));
        } else if (method != kCFD && j > 1 && j < N - 1) {
            acc = mulr((T)mim_w(0), ul[(j - 1) * es]);
#pragma unroll
            for (int i = 1; i < 4; ++i) acc = fmar((T)mim_w(i), ul[(j - 1 + i) * es], acc);
        } else {
            double w[6];
            int c0 = 0;
            const int n = method == kCFD ? cfd_Q_row(N, j, &c0, w) : mfd_G_row(N, j, &c0, w);
            for (int i = 0; i < n; ++i) acc = fmar((T)w[i], ul[(c0 + i) * es], acc);
        }
        x[l * pitch + j] = mulr(acc, ih);
    }
    __syncthreads();
    if (method == kCFD) {
        if ((int)threadIdx.x < sh.nl) fp_thomas<T>(x + threadIdx.x * pitch, N + 1, P);
        __syncthreads();
    }
}

// Dv of the share's velocity lines v: CFD Pbar^{-1} Qbar / h at nodes 1..N-1; MFD D4 / h at cells 1..N.  Into x[l *
// pitch + k], k the pressure index.
template <typename T>
__device__ void fp_dv(int method, int N, T ih, const T *v, long long ls, long long es, const FpShare &sh, T *x, int pitch,
                      FpTri<T> Pb) {
    const int l = sh.line(es == 1), last = method == kCFD ? N - 1 : N;
    const T *vl = v + (sh.line0 + l) * ls;
    for (int k = 1 + sh.first(es == 1); k <= last && l < sh.nl; k += sh.step()) {
        T acc = T(0);
        if (method == kCFD && k > 1 && k < N - 1) {
            acc = fmar(T(3), vl[(k + 1) * es], mulr(T(-3), vl[(k - 1) * es]));
        } else if (method != kCFD && k > 1 && k < N) {
            acc = mulr((T)mim_w(0), vl[(k - 2) * es]);
#pragma unroll
            for (int i = 1; i < 4; ++i) acc = fmar((T)mim_w(i), vl[(k - 2 + i) * es], acc);
        } else {
            double w[6];
            int c0 = 0;
            const int n = method == kCFD ? cfd_Qbar_row(N, k, &c0, w) : mfd_D_row(N, k - 1, &c0, w);
            for (int i = 0; i < n; ++i) acc = fmar((T)w[i], vl[(c0 + i) * es], acc);
        }
        x[l * pitch + k] = mulr(acc, ih);
    }
    __syncthreads();
    if (method == kCFD) {  // Pbar's rows 0 .. N-2 are the nodes 1 .. N-1
        if ((int)threadIdx.x < sh.nl) fp_thomas<T>(x + threadIdx.x * pitch + 1, N - 1, Pb);
        __syncthreads();
    }
}
__host__ __device__ inline int fp_pitch(int N) { return (N + 2) | 1; }

// Explicit right-hand side of a stage along its explicit direction:
//   ov = vl - beta Du(ul)   (all N+1 velocities),   oa = ul - alpha Dv(vl)   (interior)
// ul0 / ul1 (and vl0 / vl1): the iterate's buffers, picked by the parity of st->k (st may be null).
template <typename T>
__global__ void __launch_bounds__(kFpThreads) fp_rhs_kernel(int method, FpLines g, T ih, T beta, const T *ul0, const T *ul1,
                                                            const T *vl0, const T *vl1, const T *__restrict__ alpha, T *ov,
                                                            T *oa, FpTri<T> P, FpTri<T> Pb, const FpState *st, int lines) {
    extern __shared__ __align__(16) unsigned char fp_smem[];
    T *x = (T *)fp_smem;
    const bool odd = st && (st->k & 1);
    const T *ul = odd ? ul1 : ul0, *vl = odd ? vl1 : vl0;
    const FpShare sh(g, lines);
    const int pitch = fp_pitch(g.N), l = sh.line(g.esv == 1);
    fp_du<T>(method, g.N, ih, ul, g.lsp, g.esp, sh, x, pitch, P);
    for (int k = sh.first(g.esv == 1); k <= g.N && l < sh.nl; k += sh.step()) {
        const long long o = (sh.line0 + l) * g.lsv + k * g.esv;
        ov[o] = fmar(-beta, x[l * pitch + k], vl[o]);
    }
    __syncthreads();
    fp_dv<T>(method, g.N, ih, vl, g.lsv, g.esv, sh, x, pitch, Pb);
    for (int k = 1 + sh.first(g.esp == 1); k < g.L && l < sh.nl; k += sh.step()) {
        const long long o = (sh.line0 + l) * g.lsp + k * g.esp;
        oa[o] = fmar(-alpha[o], x[l * pitch + k], ul[o]);
    }
}

// x - y exactly as FP64 gives it, with one FP64 conversion where FP32 already holds it (two values within a factor of
// two of each other; Knuth's two-sum finds what is left otherwise): the FP64 pipe is far slower than FP32's.
__device__ __forceinline__ double fp_diff(double x, double y) { return x - y; }
__device__ __forceinline__ double fp_diff(float x, float y) {
    const float d = __fsub_rn(x, y), yv = __fsub_rn(x, d), xv = __fadd_rn(d, yv);
    const float rest = __fadd_rn(__fsub_rn(x, xv), __fsub_rn(yv, y));
    double e = (double)d;
    if (rest != 0.f) e += (double)rest;
    return e;
}

// One sweep of Eq. 9 along the implicit direction, from the iterate (u_k, v_k) of the parity of st->k
// to the other buffers:
//   u_{k+1} = a - alpha Dv(v_k)   (interior; the end values are the Dirichlet data, in both buffers),
//   v_{k+1} = vb - beta Du(u_{k+1}),
// with the squared norms of the two updates; the last block to finish does the stopping test (the
// paper's: the sum of the two Frobenius norms against eps, or kmax sweeps).
template <typename T>
__global__ void __launch_bounds__(kFpThreads) fp_sweep_kernel(int method, FpLines g, T ih, T beta, const T *__restrict__ a,
                                                              T *u0, T *u1, T *v0, T *v1, const T *__restrict__ vb,
                                                              const T *__restrict__ alpha, FpTri<T> P, FpTri<T> Pb,
                                                              FpState *st, double eps, int kmax, int lines) {
    if (st->done) return;
    extern __shared__ __align__(16) unsigned char fp_smem[];
    T *x = (T *)fp_smem;
    const bool odd = st->k & 1;
    const T *uk = odd ? u1 : u0, *vk = odd ? v1 : v0;
    T *un = odd ? u0 : u1, *vn = odd ? v0 : v1;
    const FpShare sh(g, lines);
    const int pitch = fp_pitch(g.N), l = sh.line(g.esv == 1);
    double du2 = 0.0, dv2 = 0.0;
    fp_dv<T>(method, g.N, ih, vk, g.lsv, g.esv, sh, x, pitch, Pb);
    for (int k = 1 + sh.first(g.esp == 1); k < g.L && l < sh.nl; k += sh.step()) {
        const long long o = (sh.line0 + l) * g.lsp + k * g.esp;
        const T val = fmar(-alpha[o], x[l * pitch + k], a[o]);
        const double e = fp_diff(val, uk[o]);
        du2 += e * e;
        un[o] = val;
    }
    __syncthreads();  // u_{k+1} of the share's lines is read back by its other threads
    fp_du<T>(method, g.N, ih, un, g.lsp, g.esp, sh, x, pitch, P);
    for (int k = sh.first(g.esv == 1); k <= g.N && l < sh.nl; k += sh.step()) {
        const long long o = (sh.line0 + l) * g.lsv + k * g.esv;
        const T val = fmar(-beta, x[l * pitch + k], vb[o]);
        const double e = fp_diff(val, vk[o]);
        dv2 += e * e;
        vn[o] = val;
    }
    __shared__ double part[2][kFpThreads / 32];
    for (int o = 16; o > 0; o >>= 1) {
        du2 += __shfl_xor_sync(0xffffffffu, du2, o);
        dv2 += __shfl_xor_sync(0xffffffffu, dv2, o);
    }
    if ((threadIdx.x & 31) == 0) { part[0][threadIdx.x >> 5] = du2; part[1][threadIdx.x >> 5] = dv2; }
    __syncthreads();
    if (threadIdx.x != 0) return;
    du2 = dv2 = 0.0;
    for (int w = 0; w < kFpThreads / 32; ++w) { du2 += part[0][w]; dv2 += part[1][w]; }
    atomicAdd(&st->sum[0], du2);
    atomicAdd(&st->sum[1], dv2);
    __threadfence();
    if (atomicAdd(&st->arrived, 1u) + 1 != gridDim.x) return;
    __threadfence();
    const double test = sqrt(__ldcg(&st->sum[0])) + sqrt(__ldcg(&st->sum[1]));
    st->sum[0] = st->sum[1] = 0.0;
    st->arrived = 0;
    st->k += 1;
    st->sweeps += 1;
    if (test <= eps || st->k >= kmax) st->done = 1;
}

__global__ void fp_reset_kernel(FpState *st) {
    st->sum[0] = st->sum[1] = 0.0;
    st->arrived = 0;
    st->k = 0;
    st->done = 0;
}

// dst <- src0, or src1 where st (if given) ended a stage at an odd number of sweeps.
template <typename T>
__global__ void fp_copy_kernel(T *dst, const T *src0, const T *src1, size_t n, const FpState *st) {
    const T *src = st && (st->k & 1) ? src1 : src0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        dst[i] = src[i];
}

// Point source dt/2 f(t) / h^2 added to the right-hand side at (is, js).
template <typename T>
__global__ void fp_source_kernel(T *a, long long p, double scale, double amp, double f0, double td, double t) {
    a[p] = (T)((double)a[p] + scale * ricker(amp, f0, td, t));
}

// Host: Thomas factors of the App. A tridiagonal P (rows 0..N) or Pbar (rows 1..N-1).
void tri_factors(int N, bool bar, std::vector<double> &m, std::vector<double> &id, std::vector<double> &c) {
    const int n = bar ? N - 1 : N + 1;
    std::vector<double> a(n, 0.0), b(n, 0.0), s(n, 0.0);
    for (int r = 0; r < n; ++r) {
        double w[6];
        int c0 = 0;
        const int row = bar ? r + 1 : r;
        const int len = bar ? cfd_Pbar_row(N, row, &c0, w) : cfd_P_row(N, row, &c0, w);
        for (int i = 0; i < len; ++i) {
            const int col = (bar ? c0 - 1 : c0) + i;  // Pbar columns are nodes 1..N-1
            if (col == r - 1) a[r] = w[i];
            else if (col == r) b[r] = w[i];
            else if (col == r + 1) s[r] = w[i];
        }
    }
    m.assign(n, 0.0); id.assign(n, 0.0); c = s;
    double d = b[0];
    id[0] = 1.0 / d;
    for (int r = 1; r < n; ++r) {
        m[r] = a[r] / d;
        d = b[r] - m[r] * s[r - 1];
        id[r] = 1.0 / d;
    }
}

struct DevArr {
    void *p = nullptr;
    ~DevArr() { if (p) cudaFree(p); }
};

template <typename T>
int run_fixed(int method, int nx, int ny, double h, double dt, const double *c_field, double *U, double *V,
              double *W, int nsteps, double t0, const double *src, int kmax, double eps, long long *sweeps,
              double *ms_out) {
    const bool cfd = method == ADI_CFD;
    const int ru = cfd ? ny + 1 : ny + 2, cu = cfd ? nx + 1 : nx + 2;  // U shape
    const int rv = ru, cv = nx + 1;                                     // V shape
    const int rw = ny + 1, cw = cu;                                     // W shape
    const size_t nU = (size_t)ru * cu, nV = (size_t)rv * cv, nW = (size_t)rw * cw;
    const int pix = cfd ? nx - 1 : nx, piy = cfd ? ny - 1 : ny;

    // device arrays
    enum { dU, dV, dW, dAl, dA, dUs, dVs, dWs, dUk, dVk, dWk, dUn, dVn, dWn, dNum };
    const size_t sizes[dNum] = {nU, nV, nW, nU, nU, nU, nV, nW, nU, nV, nW, nU, nV, nW};
    DevArr arr[dNum], tri[12], state;
    for (int k = 0; k < dNum; ++k)
        if (cudaMalloc(&arr[k].p, sizes[k] * sizeof(T)) != cudaSuccess) { (void)cudaGetLastError(); return ADI_ENOMEM; }
    if (cudaMalloc(&state.p, sizeof(FpState)) != cudaSuccess) { (void)cudaGetLastError(); return ADI_ENOMEM; }
    auto P = [&](int k) { return (T *)arr[k].p; };
    cudaError_t e = cudaMemset(state.p, 0, sizeof(FpState));

    // inputs: fields, alpha = dt/2 c^2
    {
        std::vector<T> buf(std::max(nU, std::max(nV, nW)));
        auto up = [&](const double *x, size_t n, int k, double scale, bool sq) {
            for (size_t i = 0; i < n; ++i) buf[i] = (T)(sq ? scale * x[i] * x[i] : x[i]);
            if (e == cudaSuccess) e = cudaMemcpy(arr[k].p, buf.data(), n * sizeof(T), cudaMemcpyHostToDevice);
        };
        up(U, nU, dU, 1.0, false);
        up(V, nV, dV, 1.0, false);
        up(W, nW, dW, 1.0, false);
        up(c_field, nU, dAl, 0.5 * dt, true);
    }
    if (e == cudaSuccess) e = cudaMemset(arr[dA].p, 0, nU * sizeof(T));

    // Thomas factors for both line lengths (CFD only)
    FpTri<T> Px{}, Pbx{}, Py{}, Pby{};
    if (cfd) {
        int slot = 0;
        auto make = [&](int N, bool bar) {
            std::vector<double> m, id, c;
            tri_factors(N, bar, m, id, c);
            FpTri<T> t{};
            const T *ptr[3];
            const std::vector<double> *src3[3] = {&m, &id, &c};
            for (int q = 0; q < 3; ++q) {
                std::vector<T> tv(src3[q]->begin(), src3[q]->end());
                if (e == cudaSuccess) e = cudaMalloc(&tri[slot].p, tv.size() * sizeof(T));
                if (e == cudaSuccess) e = cudaMemcpy(tri[slot].p, tv.data(), tv.size() * sizeof(T), cudaMemcpyHostToDevice);
                ptr[q] = (const T *)tri[slot].p;
                ++slot;
            }
            t.m = ptr[0]; t.id = ptr[1]; t.c = ptr[2];
            // the run of equal factors around the middle row, in the precision that the kernels use
            const int n = (int)m.size();
            auto same = [&](int r, int k) { return (T)m[r] == (T)m[k] && (T)id[r] == (T)id[k] && (T)c[r] == (T)c[k]; };
            t.lo = t.hi = n / 2;
            while (t.hi < n - 1 && same(t.hi, n / 2)) ++t.hi;
            while (t.lo > 1 && same(t.lo - 1, n / 2)) --t.lo;
            return t;
        };
        Px = make(nx, false); Pbx = make(nx, true); Py = make(ny, false); Pby = make(ny, true);
    }
    if (e != cudaSuccess) { (void)cudaGetLastError(); return e == cudaErrorMemoryAllocation ? ADI_ENOMEM : ADI_ECUDA; }

    // lines: rows (x-lines, stage 1 implicit, stage 2 explicit) and columns
    FpLines rows{1, piy, nx, cfd ? nx : nx + 1, (long long)cu, 1, (long long)cv, 1};
    FpLines cols{1, pix, ny, cfd ? ny : ny + 1, 1, (long long)cu, 1, (long long)cw};
    const T ih = (T)(1.0 / h), beta = (T)(0.5 * dt);
    // lines per block: four, fewer where their rows would not fit shared memory beside the norms' 128 bytes (the longest
    // line, ADI_MAX_CELLS in FP64, takes 131 KB)
    constexpr size_t kSmem = 226 * 1024;
    static_assert((ADI_MAX_CELLS + 3) * sizeof(double) <= kSmem, "one line fits");
    auto lines_of = [&](const FpLines &g) {
        int n = kFpLines;
        while (n > 1 && (size_t)n * fp_pitch(g.N) * sizeof(T) > kSmem) n /= 2;
        return n;
    };
    auto smem = [&](const FpLines &g) { return (size_t)lines_of(g) * fp_pitch(g.N) * sizeof(T); };
    auto grid = [&](const FpLines &g) { return (unsigned)((g.n + lines_of(g) - 1) / lines_of(g)); };
    // the limit is the process's, not this call's: the same for every size, so that no call lowers it under another's
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fp_rhs_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fp_sweep_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e != cudaSuccess) { (void)cudaGetLastError(); return ADI_ECUDA; }
    FpState *st = (FpState *)state.p;
    auto copy = [&](int dst, int src0, int src1, size_t n, const FpState *s) {
        fp_copy_kernel<T><<<152 * 4, 256>>>(P(dst), P(src0), P(src1), n, s);
    };
    const double sscale = 0.5 * dt / (h * h);
    const long long sp = src ? (long long)src[0] * cu + (long long)src[1] : 0;

    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0);
    for (int m = 0; m < nsteps; ++m) {
        const double t = t0 + m * dt;
        // ---- stage 1: w* and a explicit along y (columns), then x-line sweeps; u* and v* alternate
        // between (Us, Vs) and (Uk, Vk), starting from u^m, v^m in the latter pair ----
        copy(dWs, dW, dW, nW, nullptr);
        copy(dUs, dU, dU, nU, nullptr);
        copy(dVs, dV, dV, nV, nullptr);
        copy(dUk, dU, dU, nU, nullptr);
        copy(dVk, dV, dV, nV, nullptr);
        fp_rhs_kernel<T><<<grid(cols), kFpThreads, smem(cols)>>>(method, cols, ih, beta, P(dU), P(dU), P(dW), P(dW), P(dAl),
                                                                 P(dWs), P(dA), Py, Pby, nullptr, lines_of(cols));
        if (src) fp_source_kernel<T><<<1, 1>>>(P(dA), sp, sscale, src[2], src[3], src[4], t);
        fp_reset_kernel<<<1, 1>>>(st);
        for (int k = 0; k < kmax; ++k)
            fp_sweep_kernel<T><<<grid(rows), kFpThreads, smem(rows)>>>(method, rows, ih, beta, P(dA), P(dUk), P(dUs), P(dVk),
                                                                       P(dVs), P(dV), P(dAl), Px, Pbx, st, eps, kmax,
                                                                       lines_of(rows));
        // ---- stage 2: v^{m+1} and C explicit along x (rows), then y-line sweeps from u* and w^m,
        // alternating between (Uk, Wk) and (Un, Wn) ----
        copy(dVn, dVk, dVs, nV, st);
        copy(dUn, dUk, dUs, nU, st);
        fp_rhs_kernel<T><<<grid(rows), kFpThreads, smem(rows)>>>(method, rows, ih, beta, P(dUk), P(dUs), P(dVk), P(dVs),
                                                                 P(dAl), P(dVn), P(dA), Px, Pbx, st, lines_of(rows));
        if (src) fp_source_kernel<T><<<1, 1>>>(P(dA), sp, sscale, src[2], src[3], src[4], t + dt);
        copy(dUk, dUn, dUn, nU, nullptr);
        copy(dWn, dWs, dWs, nW, nullptr);
        copy(dWk, dW, dW, nW, nullptr);
        fp_reset_kernel<<<1, 1>>>(st);
        for (int k = 0; k < kmax; ++k)
            fp_sweep_kernel<T><<<grid(cols), kFpThreads, smem(cols)>>>(method, cols, ih, beta, P(dA), P(dUk), P(dUn), P(dWk),
                                                                       P(dWn), P(dWs), P(dAl), Py, Pby, st, eps, kmax,
                                                                       lines_of(cols));
        copy(dU, dUk, dUn, nU, st);
        copy(dV, dVn, dVn, nV, nullptr);
        copy(dW, dWk, dWn, nW, st);
    }
    cudaEventRecord(e1);
    e = cudaEventSynchronize(e1);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (e == cudaSuccess) e = cudaGetLastError();
    FpState hs{};
    if (e == cudaSuccess) e = cudaMemcpy(&hs, state.p, sizeof(FpState), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) {
        std::vector<T> buf(std::max(nU, std::max(nV, nW)));
        auto down = [&](double *x, size_t n, int k) {
            if (e == cudaSuccess) e = cudaMemcpy(buf.data(), arr[k].p, n * sizeof(T), cudaMemcpyDeviceToHost);
            if (e == cudaSuccess)
                for (size_t i = 0; i < n; ++i) x[i] = (double)buf[i];
        };
        down(U, nU, dU);
        down(V, nV, dV);
        down(W, nW, dW);
    }
    if (e != cudaSuccess) { (void)cudaGetLastError(); return ADI_ECUDA; }
    if (sweeps) *sweeps = hs.sweeps;
    if (ms_out) *ms_out = ms;
    return ADI_OK;
}

}  // namespace
}  // namespace adi

extern "C" int adi_fixed_point(int method, int nx, int ny, double h, double dt, const double *c_field, double *u,
                               double *v, double *w, int nsteps, double t0, const double *source, int kmax,
                               double eps, int precision, long long *sweeps, double *device_ms) {
    if ((method != ADI_CFD && method != ADI_MFD) || (precision != ADI_FP32 && precision != ADI_FP64) ||
        nx < ADI_MIN_CELLS || ny < ADI_MIN_CELLS || nx > ADI_MAX_CELLS || ny > ADI_MAX_CELLS ||
        !(std::isfinite(h) && h > 0) || !(std::isfinite(dt) && dt > 0) || !c_field || !u || !v || !w ||
        nsteps < 0 || kmax < 1 || !(eps >= 0.0))
        return ADI_EINVAL;
    if (source) {
        const int piy = method == ADI_CFD ? ny - 1 : ny, pix = method == ADI_CFD ? nx - 1 : nx;
        const int is = (int)source[0], js = (int)source[1];
        if (is < 1 || is > piy || js < 1 || js > pix) return ADI_EINVAL;
    }
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) { (void)cudaGetLastError(); return ADI_ENOTSUP; }
    return precision == ADI_FP64
               ? adi::run_fixed<double>(method, nx, ny, h, dt, c_field, u, v, w, nsteps, t0, source, kmax, eps, sweeps, device_ms)
               : adi::run_fixed<float>(method, nx, ny, h, dt, c_field, u, v, w, nsteps, t0, source, kmax, eps, sweeps, device_ms);
}
