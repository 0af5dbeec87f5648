// adi_kernels.cu -- line kernels of the Peaceman-Rachford ADI step (arXiv 2006.07583,
// Sec. 2, Eqs. 6-10 and 12) for sm_103a.
//
//   precompute  FP64, once per line: eliminates the one-sided boundary rows of App. A/B
//               (head and tail of every line system) into small tables.
//   prologue    turns natural fields (u, v, w) into the carried stage-1 state
//               a = u - alpha Dbar_y w + dt/2 f and w* = w - beta D_y u (Eq. 8's A and
//               Alg. 1/2's W*).
//   line_solve  one half step on a set of lines, thread per line: builds the block
//               tridiagonal line system on the fly from alpha and the stencils, block
//               Thomas forward sweep (factors kept in a global scratch), backward sweep,
//               then the carried outputs C = 2u* - a (+ dt/2 f), v' = 2v* - v.
//   finite      NaN/Inf scan of a field.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <vector>

#include "adi_internal.h"
#include "adi_ops.cuh"
#include "adi_line.cuh"

namespace adi {

// Head and tail elimination tables, one warp per (line, end): the entries of the eliminated rows, their
// inverse and the products spread over the lanes.  (One thread per line took 221 us for the 126 lines of a
// 64 x 64 grid, a chain of some 150 evaluated entries and two 5 x 5 inversions each; this 14 us.)
constexpr int kTabWarps = 4;
template <typename T>
__global__ void __launch_bounds__(32 * kTabWarps) precompute_kernel(const LineDesc<T> *__restrict__ descs, int nlines,
                                                                    T *tab_out_base, int *status) {
    __shared__ double ws[kTabWarps][4 * 36];
    const int lane = threadIdx.x & 31, job = blockIdx.x * kTabWarps + (threadIdx.x >> 5), line = job >> 1, end = job & 1;
    if (line >= nlines) return;
    const LineDesc<T> &d = descs[line];
    const LineShape s = line_shape(d.method, d.N);
    T *t = tab_out_base + (size_t)line * kTabLine + end * kTabEnd;
    const int bs = s.bs;
    const int m = end == 0 ? s.hu : s.tu;
    // index ranges: region R (the m eliminated unknowns), adjacent block J (bs)
    const int r0 = end == 0 ? 0 : s.nunk - s.tu;
    const int j0 = end == 0 ? s.hu : s.nunk - s.tu - bs;
    double *H = ws[threadIdx.x >> 5], *Hi = H + 36, *E = Hi + 36, *F = E + 18, *HiE = F + 18;
    for (int i = lane; i < m * m; i += 32) H[i] = line_entry(d, r0 + i / m, r0 + i % m);
    for (int i = lane; i < m * bs; i += 32) E[i] = line_entry(d, r0 + i / bs, j0 + i % bs);
    for (int i = lane; i < bs * m; i += 32) F[i] = line_entry(d, j0 + i / m, r0 + i % m);
    __syncwarp();
    if (!warp_inverse(H, m, Hi, lane)) {
        if (lane == 0) atomicExch(status, 1);
        return;
    }
    for (int i = lane; i < m * m; i += 32) t[kTabHinv + i] = (T)Hi[i];
    for (int i = lane; i < m * bs; i += 32) {
        double acc = 0.0;
        for (int k = 0; k < m; ++k) acc += Hi[(i / bs) * m + k] * E[k * bs + i % bs];
        HiE[i] = acc;
        t[kTabHinvE + i] = (T)acc;
    }
    for (int i = lane; i < bs * m; i += 32) {
        double acc = 0.0;
        for (int k = 0; k < m; ++k) acc += F[(i / m) * m + k] * Hi[k * m + i % m];
        t[kTabK + i] = (T)acc;
    }
    __syncwarp();
    for (int i = lane; i < bs * bs; i += 32) {
        double acc = 0.0;
        for (int k = 0; k < m; ++k) acc += F[(i / bs) * m + k] * HiE[k * bs + i % bs];
        t[kTabDB + i] = (T)acc;
    }
}

// ---------------------------------------------------------------------------------------
// Thread-per-line solver.
// ---------------------------------------------------------------------------------------
__host__ __device__ inline int v1_words(const LineShape &s) { return s.nunk + s.nb * (s.bs * s.bs + s.bs); }
size_t v1_scratch_words(int method, int N) { return (size_t)v1_words(line_shape(method, N)); }

// LANES = 1: one thread, its scratch in global memory with stride st.  LANES = 32: one warp whose line is staged
// in shared memory (L), with unit stride; the two sweeps are lane 0's, everything else is spread over the lanes.
template <typename T, int BS, int LANES>
__device__ void solve_line_v1(const LineDesc<T> &d, const Line<T> &L, T *scr, long long st, int lane, int write_natural) {
    const LineShape s = line_shape(d.method, d.N);
    const int N = d.N, hu = s.hu, tu = s.tu, nb = s.nb, nunk = s.nunk;
    auto X = [&](int k) -> T & { return scr[(long long)k * st]; };
    auto Gm = [&](int b, int i, int j) -> T & { return scr[(long long)(nunk + (b * BS + i) * BS + j) * st]; };
    auto Y = [&](int b, int i) -> T & { return scr[(long long)(nunk + nb * BS * BS + b * BS + i) * st]; };
    const T *th = d.tab, *tt = d.tab + kTabEnd;

    // right-hand sides of the two end regions
    T reg[LANES == 1 ? 12 : 1];
    T *rH = LANES == 1 ? reg : scr + v1_words(s), *rT = rH + 6;
    if constexpr (LANES == 1) {
        for (int i = 0; i < hu; ++i) rH[i] = rhs_row(L, i);
        for (int i = 0; i < tu; ++i) rT[i] = rhs_row(L, nunk - tu + i);
    } else {
        if (lane < hu) rH[lane] = rhs_row(L, lane);
        if (lane >= 16 && lane - 16 < tu) rT[lane - 16] = rhs_row(L, nunk - tu + lane - 16);
        __syncwarp();
    }

    if (lane == 0) {
    // forward sweep
    T Gp[BS][BS], yp[BS];
#pragma unroll
    for (int i = 0; i < BS; ++i) { yp[i] = T(0); for (int j = 0; j < BS; ++j) Gp[i][j] = T(0); }
    for (int b = 0; b < nb; ++b) {
        T A[BS][BS], B[BS][BS], C[BS][BS], r[BS];
        middle_block<T, T, BS>(L, s, b, A, B, C, r);
        if (b == 0) {
            for (int i = 0; i < BS; ++i) {
                for (int j = 0; j < BS; ++j) B[i][j] -= th[kTabDB + i * BS + j];
                T acc = T(0);
                for (int k = 0; k < hu; ++k) acc += th[kTabK + i * hu + k] * rH[k];
                r[i] -= acc;
            }
        }
        if (b == nb - 1) {
            for (int i = 0; i < BS; ++i) {
                for (int j = 0; j < BS; ++j) B[i][j] -= tt[kTabDB + i * BS + j];
                T acc = T(0);
                for (int k = 0; k < tu; ++k) acc += tt[kTabK + i * tu + k] * rT[k];
                r[i] -= acc;
            }
        }
        T S[BS][BS], Si[BS][BS];
#pragma unroll
        for (int i = 0; i < BS; ++i) {
#pragma unroll
            for (int j = 0; j < BS; ++j) {
                T acc = B[i][j];
#pragma unroll
                for (int k = 0; k < BS; ++k) acc -= A[i][k] * Gp[k][j];
                S[i][j] = acc;
            }
            T acc = r[i];
#pragma unroll
            for (int k = 0; k < BS; ++k) acc -= A[i][k] * yp[k];
            r[i] = acc;
        }
        mat_inv<T, BS>(S, Si);
#pragma unroll
        for (int i = 0; i < BS; ++i) {
#pragma unroll
            for (int j = 0; j < BS; ++j) {
                T acc = T(0);
#pragma unroll
                for (int k = 0; k < BS; ++k) acc += Si[i][k] * C[k][j];
                Gp[i][j] = acc;
                Gm(b, i, j) = acc;
            }
        }
        T yn[BS];
#pragma unroll
        for (int i = 0; i < BS; ++i) {
            T acc = T(0);
#pragma unroll
            for (int k = 0; k < BS; ++k) acc += Si[i][k] * r[k];
            yn[i] = acc;
        }
#pragma unroll
        for (int i = 0; i < BS; ++i) { yp[i] = yn[i]; Y(b, i) = yn[i]; }
    }
    // backward sweep: x_b = y_b - Gamma_b x_{b+1}
    T xn[BS];
#pragma unroll
    for (int i = 0; i < BS; ++i) xn[i] = T(0);
    for (int b = nb - 1; b >= 0; --b) {
        T x[BS];
#pragma unroll
        for (int i = 0; i < BS; ++i) {
            T acc = Y(b, i);
#pragma unroll
            for (int k = 0; k < BS; ++k) acc -= Gm(b, i, k) * xn[k];
            x[i] = acc;
        }
#pragma unroll
        for (int i = 0; i < BS; ++i) { xn[i] = x[i]; X(hu + b * BS + i) = x[i]; }
    }
    }
    if constexpr (LANES > 1) __syncwarp();
    // eliminated head/tail unknowns
    for (int i = lane; i < hu; i += LANES) {
        T acc = T(0);
        for (int k = 0; k < hu; ++k) acc += th[kTabHinv + i * hu + k] * rH[k];
        for (int k = 0; k < BS; ++k) acc -= th[kTabHinvE + i * BS + k] * X(hu + k);
        X(i) = acc;
    }
    const int lb = hu + (nb - 1) * BS;
    for (int i = lane; i < tu; i += LANES) {
        T acc = T(0);
        for (int k = 0; k < tu; ++k) acc += tt[kTabHinv + i * tu + k] * rT[k];
        for (int k = 0; k < BS; ++k) acc -= tt[kTabHinvE + i * BS + k] * X(lb + k);
        X(nunk - tu + i) = acc;
    }

    if constexpr (LANES > 1) __syncwarp();

    // source term dt/2 f(t_{m+1}) at the source point of this line
    T src = T(0);
    if (d.src_k >= 0) {
        long long m = *d.clock;
        double t1 = (double)(m + 1) * d.dt;
        src = (T)(d.src_scale * ricker(d.src_amp, d.src_f0, d.src_tdelay, t1));
        if constexpr (LANES > 1) __syncwarp();  // every lane has read the clock
        if (d.advance_clock && lane == 0) *d.clock = m + 1;
    }

    // epilogue: carried outputs (and natural outputs on request)
    const T beta = (T)d.beta;
    if (d.method == kCFD) {
        for (int j = lane; j <= N; j += LANES) {
            T g = X(cfd_idx_g(N, j));
            T vin = L.v(j);
            d.vo[j * d.svo] = vin - T(2) * beta * g;
            if (write_natural && d.w_out) d.w_out[j * d.snv] = vin - beta * g;
        }
        for (int j = 1 + lane; j <= N - 1; j += LANES) {
            T e = X(cfd_idx_e(j));
            T pin = L.p(j);
            T ae = L.al(j) * e;
            d.po[j * d.spo] = pin - T(2) * ae + (j == d.src_k ? src : T(0));
            if (write_natural && d.u_out) d.u_out[j * d.snp] = pin - ae;
        }
    } else {
        const T ih = (T)d.inv_h;
        const T p0 = L.p(0), pl = L.p(N + 1);
        for (int j = lane; j <= N; j += LANES) {
            double gw[8];
            int g0;
            int ng = mfd_G_row(N, j, &g0, gw);
            T acc = T(0);
            for (int t = 0; t < ng; ++t) {
                int k = g0 + t;  // pressure-line index
                T uk = (k == 0) ? p0 : (k == N + 1 ? pl : X(k - 1));
                acc += (T)gw[t] * uk;
            }
            T gu = acc * ih;
            T vin = L.v(j);
            d.vo[j * d.svo] = vin - T(2) * beta * gu;
            if (write_natural && d.w_out) d.w_out[j * d.snv] = vin - beta * gu;
        }
        for (int c = 1 + lane; c <= N; c += LANES) {
            T u = X(c - 1);
            T pin = L.p(c);
            d.po[c * d.spo] = T(2) * u - pin + (c == d.src_k ? src : T(0));
            if (write_natural && d.u_out) d.u_out[c * d.snp] = u;
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(128) line_solve_v1_kernel(const LineDesc<T> *__restrict__ descs,
                                                           int nlines, T *scratch, long long st,
                                                           int write_natural) {
    int line = blockIdx.x * blockDim.x + threadIdx.x;
    if (line >= nlines) return;
    const LineDesc<T> d = descs[line];
    T *scr = scratch + line;
    const Line<T> L(d);
    if (d.method == kCFD)
        solve_line_v1<T, 2, 1>(d, L, scr, st, 0, write_natural);
    else
        solve_line_v1<T, 3, 1>(d, L, scr, st, 0, write_natural);
}

// Short lines (at most kV1ShortCells cells): one warp per line, the line and the factors in shared memory.  So few
// lines leave the GPU idle and each is a chain of dependent steps; with a thread per line every step of
// the chain waits for global memory (64 lines of 64 cells 71 us, this 14 us).
template <typename T>
__global__ void __launch_bounds__(32) line_solve_short_kernel(const LineDesc<T> *__restrict__ descs, int write_natural) {
    extern __shared__ __align__(16) unsigned char v1_smem[];
    const LineDesc<T> &d = descs[blockIdx.x];
    const int lane = threadIdx.x, N = d.N, np = p_last(d.method, N) + 1;
    T *P = (T *)v1_smem, *Al = P + np, *V = Al + np, *scr = V + N + 1;
    for (int k = lane; k < np; k += 32) {
        P[k] = d.p[k * d.sp];
        Al[k] = d.alpha[k * d.sp];
    }
    for (int k = lane; k <= N; k += 32) V[k] = d.v[k * d.sv];
    __syncwarp();
    const Line<T> L(d, P, V, Al);
    if (d.method == kCFD)
        solve_line_v1<T, 2, 32>(d, L, scr, 1, lane, write_natural);
    else
        solve_line_v1<T, 3, 32>(d, L, scr, 1, lane, write_natural);
}

// ---------------------------------------------------------------------------------------
// Prologue: carried state from natural fields, along the stage-2 (y) lines.
//   a_k  = u_k - alpha_k (Dv w)_k + dt/2 f(t_m)   (interior pressure points) -> a
//   w*_j = w_j - beta (Du u)_j                      (all velocity points)     -> d.v
// (a is the row-major stage-1 input; d.v is the stage-2 input; the natural u and w are read through d.u_out
// and d.w_out.)
// CFD derivatives solve Pbar e = Qbar w and P g = Q u by the Thomas algorithm, with the
// factors of the two constant matrices precomputed (fac: P's sub-diagonal, eliminated
// super-diagonal and inverse pivots, N+1 each, then Pbar's, N-1 each).
// Spread over the lines' elements: prologue_mfd_kernel: MFD, block (32 lines, 8
// elements).  prologue_cfd_kernel: CFD, the two Thomas solves with the precomputed factors, one thread
// per chunk of a line, the right-hand sides formed as the sweeps need them.
// ---------------------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T prologue_src(const LineDesc<T> &d) {
    return (T)(d.src_scale * ricker(d.src_amp, d.src_f0, d.src_tdelay, (double)(*d.clock) * d.dt));
}

// Interior rows of MFD's explicit operators (D4 and G4: the fourth-order staggered stencil), with the
// weights as compile-time constants of T; the same
// terms in the same order as the row functions give them, so the sums are the same.  p points
// at the row's first point, s is the stride along the line.
template <typename T>
__device__ __forceinline__ T mfd_interior_dot(const T *p, long long s) {
    T acc = T(0);
    acc += T(1.0 / 24.0) * p[0];
    acc += T(-9.0 / 8.0) * p[s];
    acc += T(9.0 / 8.0) * p[2 * s];
    acc += T(-1.0 / 24.0) * p[3 * s];
    return acc;
}

template <typename T>
__global__ void prologue_mfd_kernel(const LineDesc<T> *__restrict__ descs, int nlines, int N, const T *__restrict__ al,
                                    int ald, T *__restrict__ a, int lda) {
    // block (32 lines, 8): elements j0 .. j0 + 31 of 32 consecutive lines; lane = line reads the
    // row-major natural fields and alpha and writes the row-major a coalesced; w*, which is contiguous along each
    // line, is written through shared memory, along each line in turn.
    __shared__ T tv[32][33], tp[32][33], tu[32][33];
    // the block's 32 descriptors, copied once with 16-byte loads (each thread would otherwise
    // read its own descriptor's fields, 32 scattered sectors per load)
    __shared__ __align__(16) unsigned char sdesc[32 * sizeof(LineDesc<T>)];
    static_assert(sizeof(LineDesc<T>) % 16 == 0, "descriptor size");
    const int x = threadIdx.x, y = threadIdx.y;
    const int line0 = blockIdx.x * 32, line = line0 + x;
    const int j0 = blockIdx.y * 32;
    {
        const int nl = min(32, nlines - line0);
        const uint4 *src = reinterpret_cast<const uint4 *>(descs + line0);
        uint4 *dst = reinterpret_cast<uint4 *>(sdesc);
        const int nvec = nl * (int)(sizeof(LineDesc<T>) / 16);
        for (int k = y * 32 + x; k < nvec; k += 256) dst[k] = src[k];
    }
    __syncthreads();
    const LineDesc<T> *sd = reinterpret_cast<const LineDesc<T> *>(sdesc);
    if (line < nlines) {
        const LineDesc<T> &d = sd[x];
        const T ih = (T)d.inv_h, beta = (T)d.beta;
        const T *un = d.u_out, *wn = d.w_out;
        const long long snp = d.snp, snv = d.snv;
        double w[8];
        int c0;
        for (int jj = y; jj < 32; jj += 8) {
            const int j = j0 + jj;
            if (j > N + 1) break;
            if (j <= N) {
                T acc = T(0);
                if (j >= 2 && j <= N - 2) {
                    acc = mfd_interior_dot(un + (long long)(j - 1) * snp, snp);
                } else {
                    const int n = mfd_G_row(N, j, &c0, w);
                    for (int t = 0; t < n; ++t) acc += (T)w[t] * un[(c0 + t) * snp];
                }
                tv[jj][x] = wn[j * snv] - beta * acc * ih;
            }
            tu[jj][x] = un[j * snp];
            if (j >= 1 && j <= N) {
                // a = u - alpha (D w)/h (+ source), formed below
                T acc = T(0);
                if (j >= 2 && j <= N - 1) {
                    acc = mfd_interior_dot(wn + (long long)(j - 2) * snv, snv);
                } else {
                    const int n = mfd_D_row(N, j - 1, &c0, w);
                    for (int t = 0; t < n; ++t) acc += (T)w[t] * wn[(c0 + t) * snv];
                }
                tp[jj][x] = acc;
            }
        }
    }
    __syncthreads();
    // w*, lane = element: 8 lines at a time, 32 consecutive elements each
    for (int l = y; l < 32 && line0 + l < nlines; l += 8) {
        const LineDesc<T> &dl = sd[l];
        const int j = j0 + x;
        if (j <= N) dl.v[(long long)j * dl.sv] = tv[x][l];
    }
    // a, lane = line
    if (line >= nlines) return;
    const LineDesc<T> &d = sd[x];
    for (int jj = y; jj < 32; jj += 8) {
        const int j = j0 + jj;
        if (j > N + 1) break;
        T val = tu[jj][x];  // j = 0 or N+1: Dirichlet, u itself
        if (j >= 1 && j <= N) {
            val = val - al[(long long)j * ald + line] * tp[jj][x] * (T)d.inv_h;
            if (j == d.src_k) val += prologue_src(d);
        }
        a[(long long)j * lda + line] = val;
    }
}

// The two Thomas solves spread over chunks of kProR rows of every line, one thread per
// (line, chunk): a line of 4097 rows gives 65 threads instead of one, so the solve is no longer a
// chain of thousands of dependent steps per thread.  Each thread solves the rows of its chunk
// plus a halo of kProH rows on each side that are not at a line end, with the values beyond the
// halo taken as zero.  Away from the two boundary rows P and Pbar are tridiag(1, 4, 1), whose
// inverse decays by a factor 2 - sqrt(3) = 0.268 per row, so what the truncation leaves out is
// 0.268^32 = 5e-19 of the solution: the result equals the whole-line solve to rounding.  A
// window that starts inside the line eliminates from its first row as if it had no
// predecessor; those rows are interior rows, and the start-up factors of that elimination (the
// last kProH values of the factor buffer) join the whole line's factors within kProH rows.
constexpr int kProR = 64, kProH = 32, kProU = 16;  // kProU rows at a time

// Products and fused products rounded as written: the compiler may otherwise fuse a product into the sum that follows,
// or not, as the loop around it happens to be unrolled.
#ifdef __CUDA_ARCH__
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_of(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_of(double a, double b, double c) { return __fma_rn(a, b, c); }
#else
inline float mul_rn(float a, float b) { return a * b; }
inline double mul_rn(double a, double b) { return a * b; }
inline float fma_of(float a, float b, float c) { return std::fma(a, b, c); }
inline double fma_of(double a, double b, double c) { return std::fma(a, b, c); }
#endif

// One window.  rows.start(r), then rows.next(r, q) for every batch of kProU rows, gives the right-hand sides in order;
// rows.back_start(r) and rows.back(r, y) the values that out(r, x, y) takes beside the solution, from the last batch
// down.  lo, cu, id: the factors of row r0 on; su: the start-up factors.  The chunk's forward values go to tmp, those of the
// rows after it to halo (which out may overwrite).  Every batch is one trip of a rolled loop: a warp runs through
// this code once, so that straight-line code waits for its instructions, and what a batch loads is asked for a batch ahead.
// INNER: a whole chunk whose window holds no boundary row, so that the factors of all rows from r0 on are those of row r0
// (the elimination's factors settle within some 15 rows).  DIV: id and su hold the pivots and the rows divide by
// them: one rounding less a row than the product with a rounded inverse, whose error was 9 % (FP32) and 22 % (FP64) above a
// plain elimination's over lines of 16 to 128 cells; divided, 3 % below it.  For adi_step_static, whose 64 x 64 CFD step
// takes 127 us so and 121 with products.
template <bool INNER, typename T, bool DIV = false, typename Rows, typename Out>
__host__ __device__ __forceinline__ void prologue_win_rows(int n, int r0, int r1, Rows rows, const T *lo, const T *cu,
                                                           const T *id, const T *su, T *tmp, T *halo, long long ts,
                                                           Out out) {
    // The start-up forms each row from the row before's unrounded product and rounds it after every S rows.  There is no
    // numerical reason for the eight: it is how an unrolled loop was once contracted, kept so that the results are the same bits
    constexpr int U = kProU, S = 8;
    static_assert(kProH % U == 0 && kProR % U == 0 && U % S == 0, "whole batches");
    const int nr = INNER ? kProR : r1 - r0;
    const int m = INNER ? kProR + kProH : (r1 + kProH < n ? r1 + kProH : n) - r0;  // m > nr only for nr = kProR
    const T lo0 = lo[0], id0 = id[0], cu0 = cu[0];
    T q[U], dd = T(0);
    rows.start(r0 > 0 ? r0 - kProH : 0);
    if (r0 > 0) {
        T t = T(0);
#pragma unroll 1
        for (int k = 0; k < kProH; k += U) {
            rows.next(r0 - kProH + k, q);
#pragma unroll
            for (int i = 0; i < U; ++i) {
                if constexpr (DIV) {
                    dd = (q[i] - dd) / su[k + i];
                } else {
                    t = i % S == 0 ? q[i] - dd : fma_of(-t, su[k + i - 1], q[i]);
                    if (i % S == S - 1) dd = mul_rn(t, su[k + i]);
                }
            }
        }
    }
#pragma unroll 1
    for (int o = 0; o < m; o += U) {
        rows.next(r0 + o, q);
        T *to = o < kProR ? tmp + o * ts : halo + (o - kProR) * ts;
#pragma unroll
        for (int i = 0; i < U; ++i)
            if (INNER || o + i < m) {
                const T num = fma_of(-(INNER ? lo0 : lo[o + i]), dd, q[i]), f = INNER ? id0 : id[o + i];
                dd = DIV ? num / f : mul_rn(num, f);
                to[i * ts] = dd;
            }
    }
    T x = T(0);
    const int top = (m - 1) / U * U;
    rows.back_start(r0 + top);
#pragma unroll 1
    for (int o = top; o >= 0; o -= U) {
        const T *from = o < kProR ? tmp + o * ts : halo + (o - kProR) * ts;
        T f[U];
#pragma unroll
        for (int i = 0; i < U; ++i) f[i] = INNER || o + i < m ? from[i * ts] : T(0);
        rows.back(r0 + o, q);
#pragma unroll
        for (int i = U - 1; i >= 0; --i)
            if (INNER || o + i < m) {
                x = fma_of(-(INNER ? cu0 : cu[o + i]), x, f[i]);
                if (o < kProR && (INNER || o + i < nr)) out(r0 + o + i, x, q[i]);
            }
    }
}

// Whether the chunk [r0, r1) of an n-row system is INNER.
__host__ __device__ inline bool prologue_inner(int n, int r0, int r1) { return r0 > 0 && r1 + kProH < n; }

// The same with right-hand sides q(r) and out(r, x); lo, cu, id of the whole line, forward values in tmp[(r - t0) * ts].
template <typename T, typename QF>
struct ProRowsOf {
    QF q;
    int n;
    __host__ __device__ void start(int) {}
    __host__ __device__ void next(int r, T (&v)[kProU]) {
        for (int i = 0; i < kProU; ++i) v[i] = r + i < n ? q(r + i) : T(0);
    }
    __host__ __device__ void back_start(int) {}
    __host__ __device__ void back(int, T (&)[kProU]) {}
};
template <typename T, typename QF, typename Out>
__host__ __device__ __forceinline__ void prologue_win_solve(int n, int r0, int r1, QF q, const T *lo, const T *cu,
                                                            const T *id, const T *su_id, T *tmp, long long ts,
                                                            Out out, int t0 = 0) {
    prologue_win_rows<false, T>(n, r0, r1, ProRowsOf<T, QF>{q, n}, lo + r0, cu + r0, id + r0, su_id, tmp + (r0 - t0) * ts,
                         tmp + (r0 - t0 + kProR) * ts, ts, [&](int r, T x, T) { out(r, x); });
}

// The rows of the kernel below: q(r) = (3 x(r + 1) - 3 x(r - 1)) ih but for the boundary rows 0 and n - 1, x(k) for k0 <=
// k <= k1 loaded once each, and y(r).
template <typename T, bool INNER, typename P = const T *>
struct ProRows {
    P x, y;
    int xs, ys, k0, k1, n, r0, r1;
    T ih, first, last, below, at, v[kProU];
    __host__ __device__ T ld(int k) const { return x[(long long)(INNER ? k : min(max(k, k0), k1)) * xs]; }
    __host__ __device__ void start(int s) {
        below = ld(s - 1);
        at = ld(s);
#pragma unroll
        for (int i = 0; i < kProU; ++i) v[i] = ld(s + 1 + i);
    }
    __host__ __device__ void next(int r, T (&q)[kProU]) {
        T w[kProU];
        // an INNER window's last batch asks for nothing: what would come next lies up to 16 rows beyond the window and
        // is not used, and the field may end with the window's last row
        const bool more = !INNER || r + kProU < r1 + kProH;
        if (more)
#pragma unroll
            for (int i = 0; i < kProU; ++i) w[i] = ld(r + kProU + 1 + i);
#pragma unroll
        for (int i = 0; i < kProU; ++i) {
            q[i] = mul_rn(fma_of(T(3), v[i], mul_rn(T(-3), below)), ih);
            below = at;
            at = v[i];
        }
        if (more)
#pragma unroll
            for (int i = 0; i < kProU; ++i) v[i] = w[i];
        if (INNER) return;
        if (r == 0) q[0] = first;
        if (r + kProU >= n)
#pragma unroll
            for (int i = 0; i < kProU; ++i)
                if (r + i == n - 1) q[i] = last;
    }
    __host__ __device__ void back_start(int r) { ask(r); }
    __host__ __device__ void back(int r, T (&out)[kProU]) {
#pragma unroll
        for (int i = 0; i < kProU; ++i) out[i] = v[i];
        ask(r - kProU);
    }
    __host__ __device__ void ask(int r) {
        if (r < r0 || r >= r1) return;  // no batch of the chunk
#pragma unroll
        for (int i = 0; i < kProU; ++i) v[i] = y[(long long)(INNER ? r + i : min(r + i, r1 - 1)) * ys];
    }
};

// A warp takes 32 consecutive lines and one chunk of P (N+1 rows) or Pbar (N-1 rows); grid.y times the
// block's warps: the chunks of P first, then those of Pbar.  The lines' natural fields are row-major, so
// lane = line reads them coalesced, and the right-hand sides Q u / h and Qbar w / h are formed row by row
// from them instead of in a pass of its own; the two boundary rows' values are formed beforehand.  a, in the
// layout that stage 1 reads, and alpha are row-major too; w* is contiguous along each line and is written through
// shared memory, lane = row.  (a in the y-lines' layout went the same way, with a transpose after it: 20 steps and
// the read of 640 x 640 cells with absorbing layers 1042 us, now 975.)  Every value is rounded as the two-pass form
// rounded it.  Few warps are in flight, so latency and, on small grids, the first fetch of the code bound it:
// with a loop per kind of row unrolled in full and loads where they are used it took 305 us for 4096 lines of 4097
// rows, 25 for 640 of 641 and 22 for 63 of 65; now 208, 17 and 16 (the two passes 531 and 46).  Rows in batches of 8: 11 %
// slower; of 32: as 16, with spills.
template <typename T>
constexpr int kProWarps = sizeof(T) == 4 ? 2 : 1;

template <typename T, bool DIV>
__global__ void __launch_bounds__(32 * kProWarps<T>) prologue_cfd_kernel(const LineDesc<T> *__restrict__ descs, int nlines,
                                                                         int N, const T *__restrict__ fac, const T *__restrict__ al,
                                                                         int ald, T *__restrict__ a, int lda) {
    __shared__ T stile[kProWarps<T>][kProR][33];  // per line: the forward values, then the solution
    __shared__ T stu[kProWarps<T>][kProR][33];    // forward values after the chunk, then w or u at its points
    __shared__ T sfac[kProWarps<T>][3][kProR + kProH], ssu[kProWarps<T>][kProH];
    __shared__ __align__(16) unsigned char sdesc[32 * sizeof(LineDesc<T>)];
    static_assert(sizeof(LineDesc<T>) % 16 == 0, "descriptor size");
    const int lane = threadIdx.x, warp = threadIdx.y;
    const int line0 = blockIdx.x * 32, nl = min(32, nlines - line0);
    {
        const uint4 *src = reinterpret_cast<const uint4 *>(descs + line0);
        uint4 *dst = reinterpret_cast<uint4 *>(sdesc);
        const int nvec = nl * (int)(sizeof(LineDesc<T>) / 16);
        for (int k = warp * 32 + lane; k < nvec; k += 32 * kProWarps<T>) dst[k] = src[k];
    }
    __syncthreads();
    const LineDesc<T> *sd = reinterpret_cast<const LineDesc<T> *>(sdesc);
    T (*tile)[33] = stile[warp], (*tu)[33] = stu[warp];
    const int nP = N + 1, nB = N - 1;
    const int chP = (nP + kProR - 1) / kProR, chB = (nB + kProR - 1) / kProR;
    const int ch = blockIdx.y * kProWarps<T> + warp;
    if (ch >= chP + chB) return;
    const bool isP = ch < chP;
    const int c = isP ? ch : ch - chP;
    const int r0 = c * kProR, r1 = min(isP ? nP : nB, r0 + kProR), nr = r1 - r0;
    // P g = (Q u)/h over rows 0..N, w*_r = w_r - beta g_r; or Pbar e = (Qbar w)/h over nodes 1..N-1 (rows 0..N-2),
    // a_j = u_j - alpha_j e_j (+ source)
    const int n = isP ? nP : nB;
    {
        const T *f = isP ? fac : fac + 3 * nP, *su = fac + 3 * nP + 3 * nB;
        const int m = min(r1 + kProH, n) - r0;
        for (int k = lane; k < m; k += 32) {
            sfac[warp][0][k] = f[r0 + k];
            sfac[warp][1][k] = f[n + r0 + k];
            sfac[warp][2][k] = f[2 * n + r0 + k];
        }
        ssu[warp][lane] = su[lane];
    }
    __syncwarp();
    if (lane < nl) {
        const LineDesc<T> &d = sd[lane];
        const T *__restrict__ un = d.u_out, *__restrict__ wn = d.w_out;
        const int xs = (int)(isP ? d.snp : d.snv), ys = (int)(isP ? d.snv : d.snp);
        const T *x = isP ? un : wn + xs, *y = isP ? wn : un + ys;
        const int k1 = isP ? N : N - 1;
        const T ih = (T)d.inv_h;
        auto out = [&](int r, T g, T y_r) {
            tile[r - r0][lane] = g;
            tu[r - r0][lane] = y_r;
        };
        const T *lo = sfac[warp][0], *cu = sfac[warp][1], *id = sfac[warp][2], *su = ssu[warp];
        if (!DIV && prologue_inner(n, r0, r1)) {  // DIV: lines too short for one
            ProRows<T, true> rows{x, y, xs, ys, 0, k1, n, r0, r1, ih};
            prologue_win_rows<true, T>(n, r0, r1, rows, lo, cu, id, su, &tile[0][lane], &tu[0][lane], 33, out);
        } else {
            auto boundary = [&](int j) {  // the first or last row of Q or Qbar
                double w[8];
                int c0;
                const int cnt = isP ? cfd_Q_row(N, j, &c0, w) : cfd_Qbar_row(N, j, &c0, w);
                const T *b = isP ? un : wn;
                T acc = T(0);
                for (int t = 0; t < cnt; ++t) acc += (T)w[t] * b[(long long)(c0 + t) * xs];
                return mul_rn(acc, ih);
            };
            ProRows<T, false> rows{x, y, xs, ys, isP ? 0 : -1, k1, n, r0, r1, ih};
            rows.first = r0 == 0 ? boundary(isP ? 0 : 1) : T(0);
            rows.last = r1 + kProH >= n ? boundary(isP ? N : N - 1) : T(0);
            prologue_win_rows<false, T, DIV>(n, r0, r1, rows, lo, cu, id, su, &tile[0][lane], &tu[0][lane], 33, out);
        }
        if (!isP && c == 0) {
            a[line0 + lane] = un[0];
            a[(long long)N * lda + line0 + lane] = un[(long long)N * d.snp];
        }
    }
    __syncwarp();
    if (isP) {  // w*, lane = row, a line's two halves at a time
#pragma unroll 8
        for (int l = 0; l < nl; ++l) {
            const LineDesc<T> &dl = sd[l];
            T *w = dl.v + (r0 + lane) * dl.sv;
            const T beta = (T)dl.beta;
#pragma unroll
            for (int k = 0; k < kProR / 32; ++k)
                if (lane + 32 * k < nr) w[32 * k * dl.sv] = fma_of(-beta, tile[lane + 32 * k][l], tu[lane + 32 * k][l]);
        }
    } else if (lane < nl) {  // a, lane = line, some rows' loads at a time
        const LineDesc<T> &d = sd[lane];
        const T *al_r = al + (long long)(r0 + 1) * ald + line0 + lane;
        T *a_r = a + (long long)(r0 + 1) * lda + line0 + lane;
        const int src = d.src_k - (r0 + 1);
#pragma unroll 1
        for (int k = 0; k < nr; k += kProU) {
            T v[kProU];
#pragma unroll
            for (int i = 0; i < kProU; ++i) v[i] = k + i < nr ? al_r[(long long)(k + i) * ald] : T(0);
#pragma unroll
            for (int i = 0; i < kProU; ++i) {
                if (k + i >= nr) break;
                T val = fma_of(-v[i], tile[k + i][lane], tu[k + i][lane]);
                if (k + i == src) val += prologue_src(d);
                a_r[(long long)(k + i) * lda] = val;
            }
        }
    }
}

// Sets *flag if any x[i] is NaN or infinite: 16-byte loads over the aligned body of x (when x
// itself is 16-byte aligned), element loads for the rest.
template <typename T>
__global__ void finite_check_kernel(const T *__restrict__ x, size_t n, int *flag) {
    constexpr int V = 16 / sizeof(T);
    const size_t i0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const size_t nv = ((size_t)x & 15u) == 0 ? n / V : 0;
    bool bad = false;
    if constexpr (sizeof(T) == 4) {
        const float4 *xv = reinterpret_cast<const float4 *>(x);
        for (size_t i = i0; i < nv; i += stride) {
            const float4 q = xv[i];
            bad |= !(isfinite(q.x) && isfinite(q.y) && isfinite(q.z) && isfinite(q.w));
        }
    } else {
        const double2 *xv = reinterpret_cast<const double2 *>(x);
        for (size_t i = i0; i < nv; i += stride) {
            const double2 q = xv[i];
            bad |= !(isfinite(q.x) && isfinite(q.y));
        }
    }
    for (size_t i = nv * V + i0; i < n; i += stride) bad |= !isfinite((double)x[i]);
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicExch(flag, 1);
}

// ---------------------------------------------------------------------------------------
// Launchers.
// ---------------------------------------------------------------------------------------
template <typename T>
cudaError_t launch_precompute(const LineDesc<T> *d, int nlines, T *tab, int *status,
                              cudaStream_t s) {
    if (nlines <= 0) return cudaSuccess;
    const int jobs = 2 * nlines;
    precompute_kernel<T><<<(jobs + kTabWarps - 1) / kTabWarps, 32 * kTabWarps, 0, s>>>(d, nlines, tab, status);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_line_solve_v1(const LineDesc<T> *d, int nlines, T *scratch, long long st,
                                 int write_natural, cudaStream_t s) {
    if (nlines <= 0) return cudaSuccess;
    int tpb = 128;
    line_solve_v1_kernel<T><<<(nlines + tpb - 1) / tpb, tpb, 0, s>>>(d, nlines, scratch, st,
                                                                    write_natural);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_line_solve_short(const LineDesc<T> *d, int nlines, int method, int N, int write_natural, cudaStream_t s) {
    if (nlines <= 0) return cudaSuccess;
    if (N > kV1ShortCells) return cudaErrorInvalidValue;
    const size_t words = 2 * (p_last(method, N) + 1) + N + 1 + v1_scratch_words(method, N) + 12;
    line_solve_short_kernel<T><<<nlines, 32, words * sizeof(T), s>>>(d, write_natural);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_prologue_lines(const LineDesc<T> *d, int nlines, int N, int method, const T *fac, const T *al, int ald,
                                  T *a, int lda, cudaStream_t s, bool pivots) {
    if (nlines <= 0) return cudaSuccess;
    if (pivots && N > kV1ShortCells) return cudaErrorInvalidValue;
    const unsigned gx = (unsigned)((nlines + 31) / 32);
    if (method == kCFD) {
        const int chunks = (N + 1 + kProR - 1) / kProR + (N - 1 + kProR - 1) / kProR, w = kProWarps<T>;
        const dim3 grid(gx, (unsigned)((chunks + w - 1) / w)), block(32, w);
        if (pivots) prologue_cfd_kernel<T, true><<<grid, block, 0, s>>>(d, nlines, N, fac, al, ald, a, lda);
        else prologue_cfd_kernel<T, false><<<grid, block, 0, s>>>(d, nlines, N, fac, al, ald, a, lda);
    } else {
        prologue_mfd_kernel<T><<<dim3(gx, (unsigned)((N + 2 + 31) / 32)), dim3(32, 8), 0, s>>>(d, nlines, N, al, ald, a, lda);
    }
    return cudaGetLastError();
}

// Thomas factors of the App. A P (N+1 rows) and Pbar (N-1 rows), for the prologue: per matrix
// the sub-diagonal, the eliminated super-diagonal c_r = up_r / den_r and 1 / den_r (pivots: den_r), where
// den_r = di_r - lo_r c_{r-1}; built in FP64.
size_t prologue_factor_count(int N) { return (size_t)3 * (N + 1) + 3 * (N - 1) + kProH; }
void prologue_factors(int N, std::vector<double> &out) {
    out.assign(prologue_factor_count(N), 0.0);
    prologue_factors(N, out.data());
}
void prologue_factors(int N, double *out, bool pivots) {
    // start-up factors of a window that begins on an interior row (no predecessor): 1 / den_k with
    // den_0 = 4, den_k = 4 - 1 / den_{k-1}
    {
        double *su = out + 3 * (N + 1) + 3 * (N - 1), den = 4.0;
        for (int k = 0; k < kProH; ++k) {
            su[k] = pivots ? den : 1.0 / den;
            den = 4.0 - 1.0 / den;
        }
    }
    for (int bar = 0; bar < 2; ++bar) {
        const int n = bar ? N - 1 : N + 1;
        double *lo = out + (bar ? 3 * (N + 1) : 0), *cu = lo + n, *id = cu + n;
        double cprev = 0.0;
        for (int r = 0; r < n; ++r) {
            double w[8];
            int c0;
            if (bar) cfd_Pbar_row(N, r + 1, &c0, w); else cfd_P_row(N, r, &c0, w);
            double l = 0.0, di, up = 0.0;
            if (r == 0) { di = w[0]; up = w[1]; }
            else if (r == n - 1) { l = w[0]; di = w[1]; }
            else { l = w[0]; di = w[1]; up = w[2]; }
            const double den = di - l * cprev;
            lo[r] = l;
            cu[r] = up / den;
            id[r] = pivots ? den : 1.0 / den;
            cprev = cu[r];
        }
    }
}
template <typename T>
cudaError_t launch_finite_check(const T *x, size_t n, int *flag, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    size_t blocks = (n + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    finite_check_kernel<T><<<(unsigned)blocks, 256, 0, s>>>(x, n, flag);
    return cudaGetLastError();
}

#define ADI_INST(T)                                                                          \
    template cudaError_t launch_precompute<T>(const LineDesc<T> *, int, T *, int *,          \
                                              cudaStream_t);                                 \
    template cudaError_t launch_line_solve_v1<T>(const LineDesc<T> *, int, T *, long long,   \
                                                 int, cudaStream_t);                         \
    template cudaError_t launch_line_solve_short<T>(const LineDesc<T> *, int, int, int, int, cudaStream_t); \
    template cudaError_t launch_prologue_lines<T>(const LineDesc<T> *, int, int, int, const T *, const T *, int, T *, int, cudaStream_t, bool); \
    template cudaError_t launch_finite_check<T>(const T *, size_t, int *, cudaStream_t);
ADI_INST(float)
ADI_INST(double)

}  // namespace adi
