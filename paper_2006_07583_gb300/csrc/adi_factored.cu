// adi_factored.cu -- the factored line solver (default): persistent CTAs, whole lines staged
// in shared memory by bulk asynchronous copies (a two-stage mbarrier ring), uniform chunks of
// MM blocks per thread held in registers, chunks joined by segmented scans of affine maps.
//
// Line system (adi_ops.cuh): every line is  [head region | nb middle blocks | tail region]
// where the middle part is block tridiagonal (blocks A_b, B_b, C_b of size BS) and the two end
// regions hold the one-sided boundary rows of App. A/B.  Here the end regions also absorb the
// remainder of nb modulo MM, so that the middle part is exactly tact * MM blocks and every
// thread runs the same unrolled code on MM blocks with no per-block predication.
//
// FP64 precompute, once per line (time invariant, depends on alpha only):
//   * each end region is eliminated densely: its unknowns become a linear map HZ of
//     z = [p window, v window, x of the adjacent middle block], the adjacent block's right-hand
//     side gets the correction KZ z and its diagonal block the correction dB;
//   * the middle part's block LU  S_b = B_b - A_b G_{b-1},  G_b = S_b^{-1} C_b  is run once and
//     per chunk c only  S at the chunk's first block,  F_c = prod(-S_b^{-1} A_b)  and
//     H_c = prod(-G_b)  are stored.
// Per half step a thread rebuilds S_b^{-1} of its blocks from the stored S and the alpha values,
// then
//   forward   y_b = S_b^{-1}(r_b - A_b y_{b-1})  locally from y = 0; the true y entering the
//             chunk is the exclusive scan of the maps (F_c, y_end) over the chunks; correction
//             y_b += d_b, d_b = -S_b^{-1} A_b d_{b-1};
//   backward  x_b = y_b - G_b x_{b+1} locally from x = 0; the true x after the chunk is the
//             suffix scan of (H_c, x_first); correction x_b += e_b, e_b = -G_b e_{b+1};
// and writes the carried outputs C = 2u* - a (+ dt/2 f), v' = 2v* - v.  The end regions are
// evaluated cooperatively by the warp that owns the adjacent chunk.
//
// The chunk transfers decay geometrically along a line (the line systems are diagonally
// dominant in the block sense).  The precompute finds, per line, the reach R: the smallest
// number of consecutive chunk transfers whose product has infinity norm below tau (2^-40 for
// FP32 records, 2^-70 for FP64).  The scan value of chunk c is then the sequential recurrence
// over the R chunks before (after) it, read from shared memory; what it leaves out is that
// product times a true value of the solution, i.e. below tau relative to the solution.  Lines
// whose reach exceeds kFacMaxReach use the full log-depth scan of affine maps instead (the
// group's kFacOwnFull bit, set on the host from the line's own reach).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstddef>

#include "../../include/adi.h"
#include "adi_internal.h"
#include "adi_line.cuh"
#include "adi_ops.cuh"

namespace adi {

constexpr int kFacThreads = 512;              // threads per CTA: 15 compute warps and one staging warp
constexpr int kFacNarrow = 256;               // MFD in FP64, lines of at most 224 chunks: 7 compute warps (fac_narrow)
constexpr int kFacWorkers = kFacThreads - 32; // threads that solve lines
constexpr int kFacMaxT = kFacWorkers;         // chunks (threads) per line at most
constexpr size_t kFacSmemLimit = 227 * 1024;  // shared memory per CTA
constexpr size_t kFacStaticBase = 2048;       // reserve for the kernel's other static shared memory
constexpr int kFacMaxStages = 3;              // staged groups in flight per CTA at most
constexpr int kFacWs = 1024;                  // FP64 workspace of one end's elimination
// Static shared memory of the kernel for element size esz and block size bs, an upper bound:
// the scan buffers (chunk offsets, two arrays for FP32, one for FP64) plus the rest (checked
// against the compiled kernel before its first launch).
__host__ __device__ inline size_t fac_static_smem(size_t esz, int bs) {
    return kFacStaticBase + (size_t)kFacThreads * bs * (esz == 4 ? 2 : 1) * esz;
}

// One rounding for a*b + c, written out so that the compiler's contraction choices cannot make
// two code paths of the same output round differently.
#ifdef __CUDA_ARCH__
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
#else
inline float fma_rn(float a, float b, float c) { return std::fma(a, b, c); }
inline double fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
inline float mul_rn(float a, float b) { return a * b; }
inline double mul_rn(double a, double b) { return a * b; }
inline double add_rn(double a, double b) { return a + b; }
inline double sub_rn(double a, double b) { return a - b; }
#endif

// ---------------------------------------------------------------------------------------
// Geometry of a line for the factored solver.
// ---------------------------------------------------------------------------------------
// Blocks per chunk: CFD 9 (an odd stride between the chunks' shared-memory windows keeps
// their loads free of bank conflicts); MFD 3 (a chunk's record, S, F and H of 3 x 3, then costs
// 12 bytes per cell in FP32; two-block chunks cost 18 and ran a batch of 128-1024-cell lines 4 %
// slower), and 2 for lines of at most kFacMfdShort cells, whose end regions would not fit their
// tables with the remainder of three-block chunks.
constexpr int kFacMfdShort = 16;
__host__ __device__ inline int fac_mm(int method, int N) {
    if (method == kCFD) return 9;
    return N <= kFacMfdShort ? 2 : 3;
}
// Threads a whole line needs (see fac_geom): a power of two up to 32, else a multiple of 32.
__host__ __device__ inline int fac_geom_T(int method, int N) {
    const int tact = line_shape(method, N).nb / fac_mm(method, N);
    if (tact > 32) return (tact + 31) & ~31;
    int T = 1;
    while (T < tact) T <<= 1;
    return T;
}
// MFD lines of at most 224 chunks run in FP64 in CTAs of 256 threads: twice the registers a thread (the
// band form's 72 FP64 values do not fit 128 registers and spilled 0.5 KB a thread, more than the L1 beside the staged
// lines holds), and seven warps keep the FP64 pipe as busy as fifteen: 1001 lines of 1001 cells 200 ->
// 144 us with the band form; a step at 20 to 2024 cells a side 5 to 16 % faster than in wide CTAs, 1.4 % slower at 881 to 934,
// where a CTA takes one line in place of two.  CFD, whose lines of 512 cells then made two rounds instead of one, gained
// nothing (55.7 -> 58.0 us) and keeps the wide CTAs.
__host__ __device__ inline bool fac_narrow(int method, int T, size_t esz) {
    return method == kMFD && esz == 8 && T <= kFacNarrow - 32;
}
// Kernel variant (one compiled instance per chunk length and method, and for split lines).
__host__ __device__ inline int fac_variant_of(int method, int N) {
    const bool split = fac_geom_T(method, N) > kFacMaxT;
    if (method == kCFD) return split ? 3 : 0;
    return fac_mm(method, N) == 2 ? 1 : (split ? 4 : 2);
}
// End windows: p[op .. op+win) and v[ov .. ov+win); hmax bounds the eliminated unknowns of
// one end (base head/tail plus half of at most MM-1 remainder blocks).
__host__ __device__ inline int fac_win(int method) { return method == kCFD ? 8 : 12; }
__host__ __device__ inline int fac_hmax(int method) { return method == kCFD ? 13 : 8; }

struct FacGeom {
    int method, N, bs, mm;
    int hu, tu;   // eliminated unknowns of the head and tail regions
    int nb;       // middle blocks (tact * mm)
    int tact;     // chunks holding blocks
    int T;        // threads per line: a power of two up to 32, else a multiple of 32
    int first;    // CFD: node of middle block 0; MFD: first cell of middle block 0
    int win, hmax;
};

__host__ __device__ inline FacGeom fac_geom(int method, int N) {
    const LineShape s = line_shape(method, N);
    FacGeom g;
    g.method = method;
    g.N = N;
    g.bs = s.bs;
    g.mm = fac_mm(method, N);
    g.tact = s.nb / g.mm;
    const int k = s.nb - g.tact * g.mm;
    const int kh = k / 2;
    g.hu = s.hu + kh * s.bs;
    g.tu = s.tu + (k - kh) * s.bs;
    g.nb = g.tact * g.mm;
    int T = 1;
    while (T < g.tact) T <<= 1;
    g.T = g.tact > 32 ? ((g.tact + 31) & ~31) : T;
    g.first = method == kCFD ? (g.hu + 1) / 2 : g.hu + 1;
    g.win = fac_win(method);
    g.hmax = fac_hmax(method);
    return g;
}

// Per-end table: KZ [bs][2win] | HZ [hmax][Z] | DZ [hmax+2][Z] (MFD) | dB [bs][bs], Z = 2win+bs.
__host__ __device__ inline int fac_zlen(const FacGeom &g) { return 2 * g.win + g.bs; }
__host__ __device__ inline int fac_e_hz(const FacGeom &g) { return g.bs * 2 * g.win; }
__host__ __device__ inline int fac_e_dz(const FacGeom &g) { return fac_e_hz(g) + g.hmax * fac_zlen(g); }
__host__ __device__ inline int fac_e_db(const FacGeom &g) {
    return fac_e_dz(g) + (g.method == kMFD ? (g.hmax + 2) * fac_zlen(g) : 0);
}
__host__ __device__ inline int fac_e_stride(const FacGeom &g) { return (fac_e_db(g) + g.bs * g.bs + 3) & ~3; }
// Record of one line: S_first, F_c, H_c (tact blocks each, every part padded to a multiple of
// four elements so that each starts on a 16-byte boundary), the head and tail tables, then four
// values: the forward and backward reach of the windowed scans.
__host__ __device__ inline int fac_ru4(int x) { return (x + 3) & ~3; }
__host__ __device__ inline int fac_part(const FacGeom &g) { return fac_ru4(g.tact * g.bs * g.bs); }
__host__ __device__ inline int fac_chunk_elems(const FacGeom &g) { return 3 * fac_part(g); }
__host__ __device__ inline int fac_info(const FacGeom &g) { return fac_chunk_elems(g) + 2 * fac_e_stride(g); }
__host__ __device__ inline int fac_rec(const FacGeom &g) { return fac_info(g) + 4; }
// Elements of one staged line array (pressure, velocity or alpha), a multiple of four.
__host__ __device__ inline int fac_lp(int N) { return (N + 2 + 3) & ~3; }
// Shared-memory scratch of a staged line: the window parts of its end-region rows.
__host__ __device__ inline int fac_end_rows(int method) {
    return 2 * (fac_hmax(method) + (method == kMFD ? fac_hmax(method) + 2 : 0));
}
__host__ __device__ inline int fac_scratch(const FacGeom &g) { return (fac_end_rows(g.method) + 3) & ~3; }
// A staged line: pressure, velocity, alpha (fac_lp each), the record, the scratch.
__host__ __device__ inline int fac_line_elems(const FacGeom &g) { return 3 * fac_lp(g.N) + fac_rec(g) + fac_scratch(g); }

constexpr size_t kDescBytes = sizeof(LineDesc<float>);
static_assert(sizeof(LineDesc<float>) == sizeof(LineDesc<double>), "descriptor sizes differ");
static_assert(kDescBytes % 16 == 0, "descriptor size");
__host__ __device__ inline size_t fac_desc_area(int nl) { return ((size_t)nl * kDescBytes + 127) & ~(size_t)127; }
// A stage: the group's header (its fields before the base addresses, which only the staging warp reads, from global
// memory), the descriptors, then the lines.  With the whole 192-byte record staged, lines of 703-706 MFD cells went four
// instead of five to a CTA.
constexpr size_t kFacGroupBytes = offsetof(FacGroup, gp);
static_assert(kFacGroupBytes == 128 && alignof(FacGroup) == 16, "group header");
__host__ __device__ inline size_t fac_head_bytes(int nl) { return kFacGroupBytes + fac_desc_area(nl); }

size_t fac_stage_bytes(int method, int N, int nl, size_t esz) {
    size_t b = fac_head_bytes(nl) + (size_t)nl * fac_line_elems(fac_geom(method, N)) * esz;
    return (b + 127) & ~(size_t)127;
}
int fac_stages_for(size_t stage_bytes, size_t esz, int method) {
    const size_t st = fac_static_smem(esz, method == kCFD ? 2 : 3);
    for (int k = kFacMaxStages; k >= 1; --k)
        if ((size_t)k * stage_bytes + st <= kFacSmemLimit) return k;
    return 0;
}
// Lines per CTA: as many as the CTA's threads cover, fewer where a two-stage ring of them
// would not fit shared memory.
int fac_lines_per_cta(int method, int N, size_t esz) {
    const int T = fac_geom(method, N).T, workers = fac_narrow(method, T, esz) ? kFacNarrow - 32 : kFacWorkers;
    int nl = T >= workers ? 1 : workers / T;
    while (nl > 1 && fac_stages_for(fac_stage_bytes(method, N, nl, esz), esz, method) < 2) --nl;
    return nl;
}
bool fac_split_line(int method, int N) { return fac_geom(method, N).T > kFacMaxT; }
bool fac_supported(int method, int N, size_t esz) {
    const FacGeom g = fac_geom(method, N);
    if (g.tact < 1) return false;
    if (g.hu > g.hmax || g.tu > g.hmax) return false;
    if (g.T > kFacMaxT) {  // split into sub-lines (for the largest halo a split line accepts)
        FacGroup tmp[kFacMaxSplit];
        size_t sb = 0;
        return fac_split_groups(method, N, 0, kFacSplitMaxHalo, 1.0, 1.0, esz, tmp, &sb) > 0;
    }
    return fac_stages_for(fac_stage_bytes(method, N, 1, esz), esz, method) > 0;
}
size_t fac_words(int method, int N) { return (size_t)fac_rec(fac_geom(method, N)); }
int fac_chunks(int method, int N) { return fac_geom(method, N).T; }
bool fac_direct(int method, int N) { return fac_geom(method, N).T < 32; }
int fac_variant(int method, int N, size_t esz) {
    const int v = fac_variant_of(method, N);
    return fac_narrow(method, fac_geom(method, N).T, esz) ? v + 4 : v;
}
int fac_variant_method(int v) { return v == 0 || v == 3 ? kCFD : kMFD; }
size_t fac_ws_doubles() { return 18; }
static unsigned fac_tdiv(int T) {
    return T > 1 ? (unsigned)(((1ull << 32) + (unsigned long long)T - 1) / (unsigned long long)T) : 0u;
}
FacGroup fac_group_of(int method, int N, int first, int nl, double inv_h, double beta) {
    const FacGeom g = fac_geom(method, N);
    FacGroup r{};
    r.first = first; r.nl = nl; r.N = N; r.T = g.T;
    r.tact = g.tact; r.hu = g.hu; r.tu = g.tu; r.mid = g.first;
    r.lp = fac_lp(N); r.part = fac_part(g);
    r.eh = fac_chunk_elems(g); r.et = r.eh + fac_e_stride(g);
    r.info = fac_info(g); r.pl = p_last(method, N);
    r.ls = fac_line_elems(g); r.scr = 3 * r.lp + fac_rec(g);
    r.ih = inv_h; r.beta = beta; r.ihf = (float)inv_h; r.betaf = (float)beta;
    r.tdiv = fac_tdiv(g.T);
    r.c0 = 0; r.lo = 0; r.pn = r.pl + 1; r.vn = N + 1;
    r.own = (g.tact << 9) | kFacOwnHead | kFacOwnTail;
    r.sp0 = 0; r.sp1 = r.pl + 1; r.sv0 = 0; r.sv1 = N + 1;
    return r;
}

// Sub-lines of a line with more chunks than a CTA has threads.  Sub-line i owns the chunks
// [tact i / K, tact (i+1) / K) and also solves `halo` (rounded so that its first chunk is a
// multiple of four: the record parts it stages then start on 16-byte boundaries) chunks on
// each interior side.  The windowed scans of its owned chunks reach at most `halo` chunks, all
// inside its range; the halo chunks' own scan values are truncated at the range's ends and
// their outputs are not written.  Staged elements cover every stencil read of the range; the
// owned outputs are stored by bulk copies on 4-element-aligned spans and, at the ragged ends
// of a span, by the threads that compute them.
int fac_split_groups(int method, int N, int first, int halo, double inv_h, double beta, size_t esz,
                     FacGroup *out, size_t *stage_bytes) {
    const FacGeom g = fac_geom(method, N);
    if (g.tact < 1 || g.hu > g.hmax || g.tu > g.hmax || halo < 1 || halo > kFacSplitMaxHalo) return 0;
    const int B2 = g.bs * g.bs, pl = p_last(method, N);
    const int per = method == kCFD ? g.mm : 3 * g.mm;  // nodes (CFD) or cells (MFD) per chunk
    const int vsh = method == kCFD ? 0 : 1;             // MFD: a chunk's velocities start one after its cells
    int K = 2;
    while (K <= kFacMaxSplit && (g.tact + K - 1) / K + 2 * halo + 3 > kFacMaxT) ++K;
    if (K > kFacMaxSplit) return 0;
    size_t smax = 0;
    for (int i = 0; i < K; ++i) {
        const int s0 = (int)((long long)g.tact * i / K), s1 = (int)((long long)g.tact * (i + 1) / K);
        const bool head = i == 0, tail = i == K - 1;
        const int c0 = head ? 0 : ((s0 - halo) & ~3);
        const int c1 = tail ? g.tact : std::min(g.tact, s1 + halo);
        const int tl = c1 - c0;
        if (c0 < 0 || tl > kFacMaxT || tl <= 64) return 0;
        FacGroup r{};
        r.first = first; r.nl = 1; r.N = N;
        r.tact = tl; r.T = (tl + 31) & ~31;
        r.hu = g.hu; r.tu = g.tu; r.mid = g.first;
        // staged elements [lo, hi): a CFD chunk reads nodes jb-1 .. jb+mm, an MFD chunk cells
        // cb .. cb+3mm-1 and velocities cb-2 .. cb+3mm
        const int lo = head ? 0 : ((g.first + c0 * per - 2) & ~3);
        const int hp = tail ? pl + 1 : g.first + c1 * per + 1;
        const int hv = tail ? N + 1 : g.first + c1 * per + 1;
        r.lo = lo; r.pn = hp - lo; r.vn = hv - lo;
        r.lp = fac_ru4(r.pn > r.vn ? r.pn : r.vn);
        const int part = fac_ru4(tl * B2), es = fac_e_stride(g);
        r.part = part;
        int off = 3 * part;
        r.eh = head ? off : -1;
        if (head) off += es;
        r.et = tail ? off : -1;
        if (tail) off += es;
        r.info = off;
        r.pl = pl;
        r.scr = 3 * r.lp + off + 4;
        r.ls = r.scr + fac_scratch(g);
        r.ih = inv_h; r.beta = beta; r.ihf = (float)inv_h; r.betaf = (float)beta;
        r.tdiv = fac_tdiv(r.T);
        r.c0 = c0;
        r.own = (s0 - c0) | ((s1 - c0) << 9) | (head ? kFacOwnHead : 0) | (tail ? kFacOwnTail : 0) | kFacOwnSplit;
        const int p0 = head ? 0 : g.first + s0 * per, p1 = tail ? pl + 1 : g.first + s1 * per;
        const int v0 = head ? 0 : g.first + s0 * per + vsh, v1 = tail ? N + 1 : g.first + s1 * per + vsh;
        r.sp0 = fac_ru4(p0); r.sp1 = tail ? p1 : (p1 & ~3);
        r.sv0 = fac_ru4(v0); r.sv1 = tail ? v1 : (v1 & ~3);
        out[i] = r;
        const size_t sb = (fac_head_bytes(1) + (size_t)r.ls * esz + 127) & ~(size_t)127;
        if (sb > smax) smax = sb;
    }
    *stage_bytes = smax;
    return fac_stages_for(smax, esz, method) > 0 ? K : 0;
}
// Table offsets of an end region, as compile-time functions of the block size (fac_e_*).
template <int BS>
struct FacEnd {
    static constexpr int W = BS == 2 ? 8 : 12, HMAX = BS == 2 ? 13 : 8, Z = 2 * W + BS;
    static constexpr int HZ = BS * 2 * W, DZ = HZ + HMAX * Z, DB = DZ + (BS == 3 ? (HMAX + 2) * Z : 0);
};

// Reciprocals.  FP32: the hardware approximation (relative error below 2^-22).
__device__ __forceinline__ float fac_rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// FP64: the hardware approximation r0 (about 20 bits) and one step of Householder's cubic iteration, r0 (1 + e
// + e^2) with e = 1 - x r0: three FMAs against a division's ten or so operations on the FP64 pipe that bounds these kernels;
// the error left is e^3 = 2^-60 and one rounding (measured against 1 / x: at most 1 ulp).  For the pivots of MfdBand only,
// where divisions made 1001 lines of 1001 cells 299 in place of 288 us a step and the step's error against extended precision, over grids
// of 48 to 1001 cells a side, no smaller (9.38e-16, 9.33e-16 and 7.80e-16 for u, v and w with either).
__device__ __forceinline__ double fac_rcp(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = __fma_rn(-x, r, 1.0);
    return __fma_rn(r, __fma_rn(e, e, e), r);
}

// ---------------------------------------------------------------------------------------
// FP64 precompute.
// ---------------------------------------------------------------------------------------
// Right-hand side of line row i (solver index) as coefficients on the windows
// p[op .. op+W) and v[ov .. ov+W).  False if a term falls outside them.
template <typename TS>
__device__ bool fac_rhs_coeffs(const LineDesc<TS> &d, int i, int op, int ov, int W, double *cp, double *cv) {
    for (int k = 0; k < W; ++k) cp[k] = cv[k] = 0.0;
    const int N = d.N;
    const double ih = d.inv_h;
    bool ok = true;
    auto add = [&](double *w, int idx, double val) {
        if (idx < 0 || idx >= W) ok = false; else w[idx] += val;
    };
    double w[8];
    int c0, n;
    if (d.method == kCFD) {
        const bool is_g = (i == 0) || (i == 2 * N - 1) || (i % 2 == 0);
        const int node = i == 0 ? 0 : (i == 2 * N - 1 ? N : (i + 1) / 2);
        if (is_g) {
            n = cfd_Q_row(N, node, &c0, w);
            for (int t = 0; t < n; ++t) add(cp, c0 + t - op, w[t] * ih);
        } else {
            n = cfd_Qbar_row(N, node, &c0, w);
            for (int t = 0; t < n; ++t) add(cv, c0 + t - ov, w[t] * ih);
        }
        return ok;
    }
    // r_c = p_c - alpha_c/h sum_j D[c-1][j] (v_j - beta/h (G[j][0] p_0 + G[j][N+1] p_{N+1}))
    const int c = i + 1;
    const double a = (double)d.alpha[(long long)c * d.sp], bh = d.beta * ih;
    add(cp, c - op, 1.0);
    n = mfd_D_row(N, c - 1, &c0, w);
    for (int t = 0; t < n; ++t) {
        const int node = c0 + t;
        const double coef = -a * ih * w[t];
        add(cv, node - ov, coef);
        if (node <= 1 || node >= N - 1) {
            double gw[8];
            int g0;
            const int ng = mfd_G_row(N, node, &g0, gw);
            if (g0 == 0) add(cp, 0 - op, -coef * bh * gw[0]);
            if (g0 + ng - 1 == N + 1) add(cp, N + 1 - op, -coef * bh * gw[ng - 1]);
        }
    }
    return ok;
}

// Dense elimination of one end region (end 0: head, 1: tail) into its table by one warp, in its
// shared workspace ws (kFacWs doubles); dB of the end (bs x bs, row-major) is also returned in FP64
// in dBo (global memory).  False if the region is singular.
template <typename TS>
__device__ bool fac_end(const LineDesc<TS> &d, const FacGeom &g, int end, double *ws, TS *et, double *dBo, int lane) {
    const int N = d.N, bs = g.bs, W = g.win, Z = fac_zlen(g);
    const int nunk = d.method == kCFD ? 2 * N : N;
    const int m = end == 0 ? g.hu : g.tu;
    const int r0 = end == 0 ? 0 : nunk - g.tu;
    const int j0 = end == 0 ? g.hu : nunk - g.tu - bs;
    const int pl = p_last(d.method, N);
    const int op = end == 0 ? 0 : pl + 1 - W, ov = end == 0 ? 0 : N + 1 - W;
    double *H = ws, *Hi = H + m * m, *E = Hi + m * m, *F = E + m * bs, *Rm = F + bs * m;
    double *HiE = Rm + m * 2 * W, *K = HiE + m * bs, *HZ = K + bs * m;
    for (int i = lane; i < m * m; i += 32) H[i] = line_entry(d, r0 + i / m, r0 + i % m);
    for (int i = lane; i < m * bs; i += 32) E[i] = line_entry(d, r0 + i / bs, j0 + i % bs);
    for (int i = lane; i < bs * m; i += 32) F[i] = line_entry(d, j0 + i / m, r0 + i % m);
    bool ok = true;
    if (lane < m) ok = fac_rhs_coeffs(d, r0 + lane, op, ov, W, Rm + lane * 2 * W, Rm + lane * 2 * W + W);
    ok = __all_sync(0xffffffffu, ok);
    __syncwarp();
    if (!warp_inverse(H, m, Hi, lane)) return false;
    for (int i = lane; i < m * bs; i += 32) {
        double acc = 0.0;
        for (int k = 0; k < m; ++k) acc += Hi[(i / bs) * m + k] * E[k * bs + i % bs];
        HiE[i] = acc;
    }
    for (int i = lane; i < bs * m; i += 32) {
        double acc = 0.0;
        for (int k = 0; k < m; ++k) acc += F[(i / m) * m + k] * Hi[k * m + i % m];
        K[i] = acc;
    }
    const double nan = __longlong_as_double(0x7ff8000000000000ULL);
    const int e_stride = fac_e_stride(g);
    for (int i = lane; i < e_stride; i += 32) et[i] = (TS)0;
    __syncwarp();
    for (int i = lane; i < bs * bs; i += 32) {
        double acc = 0.0;
        for (int k = 0; k < m; ++k) acc += F[(i / bs) * m + k] * HiE[k * bs + i % bs];
        dBo[i] = acc;
        et[fac_e_db(g) + i] = (TS)acc;
    }
    // KZ = -K R
    for (int i = lane; i < bs * 2 * W; i += 32) {
        double acc = 0.0;
        for (int q = 0; q < m; ++q) acc -= K[(i / (2 * W)) * m + q] * Rm[q * 2 * W + i % (2 * W)];
        et[i] = (TS)(ok ? acc : nan);
    }
    // HZ = [Hinv R | -Hinv E]
    for (int i = lane; i < m * Z; i += 32) {
        const int q = i / Z, k = i % Z;
        double acc = 0.0;
        if (k < 2 * W) {
            for (int q2 = 0; q2 < m; ++q2) acc += Hi[q * m + q2] * Rm[q2 * 2 * W + k];
        } else {
            acc = -HiE[q * bs + k - 2 * W];
        }
        HZ[i] = acc;
        et[fac_e_hz(g) + i] = (TS)(ok ? acc : nan);
    }
    __syncwarp();
    if (d.method != kMFD) return true;
    // MFD: h (G u)_j at the end's velocity nodes as maps of z (cells through HZ), lane = entry of z
    const int qb = g.first + 3 * (g.nb - 1);  // first cell of the last middle block
    const int jlo = end == 0 ? 0 : qb + 1, jhi = end == 0 ? g.hu + 1 : N;
    const int cell_lo = end == 0 ? 1 : N - g.tu + 1;  // first eliminated cell
    const int adj = end == 0 ? g.hu + 1 : qb;         // first cell of the adjacent block
    for (int j = jlo; j <= jhi; ++j) {
        double gw[8], row = 0.0;
        int g0;
        const int ng = mfd_G_row(N, j, &g0, gw);
        bool rok = ok;
        for (int t = 0; t < ng; ++t) {
            const int cc = g0 + t;
            if (cc == 0 || cc == N + 1) {
                const int wi = cc - op;
                if (wi < 0 || wi >= W) rok = false; else if (lane == wi) row += gw[t];
            } else if (cc >= cell_lo && cc < cell_lo + m) {
                if (lane < Z) row += gw[t] * HZ[(cc - cell_lo) * Z + lane];
            } else if (cc >= adj && cc < adj + bs) {
                if (lane == 2 * W + cc - adj) row += gw[t];
            } else {
                rok = false;
            }
        }
        if (lane < Z) et[fac_e_dz(g) + (j - jlo) * Z + lane] = (TS)(rok ? row : nan);
    }
    return true;
}

// The end tables: one warp per (line, end).  With one thread per line and its workspace in global memory
// the eliminations were a chain of scattered accesses and most of the 15.4 ms that the records of a
// 4096 x 4096 grid took.
constexpr int kFacEndWarps = 4;
template <typename TS>
__global__ void __launch_bounds__(32 * kFacEndWarps) fac_ends_kernel(const LineDesc<TS> *__restrict__ descs, int nlines,
                                                                     double *dB, int *status) {
    __shared__ double ws[kFacEndWarps][kFacWs];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int job = blockIdx.x * kFacEndWarps + warp, line = job >> 1, end = job & 1;
    if (line >= nlines) return;
    const LineDesc<TS> &d = descs[line];
    const FacGeom g = fac_geom(d.method, d.N);
    TS *et = d.sep + fac_chunk_elems(g) + end * fac_e_stride(g);
    if (!fac_end(d, g, end, ws[warp], et, dB + (size_t)job * 9, lane) && lane == 0) atomicExch(status, 1);
}

// Block LU of the middle blocks [b0, b1) of a line (whole chunks), from G = G_{b0-1}; on return G =
// G_{b1-1}.  STORE: write the chunks' records.  False if a block is singular.  The FP64 pipe bounds it (one
// warp instruction in 19 cycles an SM), so the products visit the coupling blocks' nonzero entries only and none
// of their units (the blocks as in fac_group); each sum keeps the order and the roundings of the full block products,
// so that leaving entries out changes no bit.
__host__ __device__ __forceinline__ bool fac_pivot_ok(double det) { return fabs(det) > 0.0 && isfinite(det); }

template <typename TS, bool STORE>
__host__ __device__ bool fac_run(const LineDesc<TS> &d, const FacGeom &g, const double *dBh, const double *dBt, TS *rec, int b0,
                        int b1, double (&G)[2][2]) {
    TS *recS = rec, *recF = rec + fac_part(g), *recH = rec + (size_t)2 * fac_part(g);
    const double tb = 3.0 * d.beta * d.inv_h, c3 = 3.0 * d.inv_h;
    const TS *__restrict__ al = d.alpha;
    const long long sp = d.sp;
    const int j0 = g.first;
    double am = c3 * (double)al[(j0 + b0 - 1) * sp], a0 = c3 * (double)al[(j0 + b0) * sp];
    double F[2][2] = {}, H[2][2] = {};
    int c = b0 / g.mm, i = 0;
    for (int b = b0; b < b1; ++b) {
        const double ap = c3 * (double)al[(j0 + b + 1) * sp];
        const bool first = b == 0, last = b == g.nb - 1;
        double S[2][2] = {{4.0, 0.0}, {0.0, 4.0}};
        if (first)
            for (int p = 0; p < 2; ++p)
                for (int q = 0; q < 2; ++q) S[p][q] -= dBh[p * 2 + q];
        if (last)
            for (int p = 0; p < 2; ++p)
                for (int q = 0; q < 2; ++q) S[p][q] -= dBt[p * 2 + q];
        if (!first) {  // S -= A G, A = [[1, -tb], [-am, 1]]
            S[0][0] = fma_rn(tb, G[1][0], sub_rn(S[0][0], G[0][0]));
            S[0][1] = fma_rn(tb, G[1][1], sub_rn(S[0][1], G[0][1]));
            S[1][0] = sub_rn(fma_rn(am, G[0][0], S[1][0]), G[1][0]);
            S[1][1] = sub_rn(fma_rn(am, G[0][1], S[1][1]), G[1][1]);
        }
        const double det = S[0][0] * S[1][1] - S[0][1] * S[1][0];
        if (!fac_pivot_ok(det)) return false;
        double R[2][2];
        mat_inv<double, 2>(S, R);
        // G = R C, C = [[1, tb], [ap, 1]]
        G[0][0] = last ? 0.0 : fma_rn(R[0][1], ap, R[0][0]);
        G[0][1] = last ? 0.0 : add_rn(mul_rn(R[0][0], tb), R[0][1]);
        G[1][0] = last ? 0.0 : fma_rn(R[1][1], ap, R[1][0]);
        G[1][1] = last ? 0.0 : add_rn(mul_rn(R[1][0], tb), R[1][1]);
        if constexpr (STORE) {
            // E = -R A
            double E[2][2] = {{-fma_rn(R[0][1], -am, R[0][0]), -add_rn(mul_rn(R[0][0], -tb), R[0][1])},
                              {-fma_rn(R[1][1], -am, R[1][0]), -add_rn(mul_rn(R[1][0], -tb), R[1][1])}};
            if (first) E[0][0] = E[0][1] = E[1][0] = E[1][1] = 0.0;
            if (i == 0) {
                for (int p = 0; p < 2; ++p)
                    for (int q = 0; q < 2; ++q) {
                        recS[(size_t)c * 4 + p * 2 + q] = (TS)S[p][q];
                        F[p][q] = E[p][q];
                        H[p][q] = -G[p][q];
                    }
            } else {
                double f[2][2], h[2][2];
                for (int p = 0; p < 2; ++p)
                    for (int q = 0; q < 2; ++q) {
                        f[p][q] = fma_rn(E[p][1], F[1][q], mul_rn(E[p][0], F[0][q]));
                        h[p][q] = -fma_rn(H[p][1], G[1][q], mul_rn(H[p][0], G[0][q]));
                    }
                for (int p = 0; p < 2; ++p)
                    for (int q = 0; q < 2; ++q) { F[p][q] = f[p][q]; H[p][q] = h[p][q]; }
            }
            if (++i == g.mm) {
                for (int p = 0; p < 2; ++p)
                    for (int q = 0; q < 2; ++q) {
                        recF[(size_t)c * 4 + p * 2 + q] = (TS)F[p][q];
                        recH[(size_t)c * 4 + p * 2 + q] = (TS)H[p][q];
                    }
                i = 0;
                ++c;
            }
        }
        am = a0;
        a0 = ap;
    }
    return true;
}

template <typename TS, bool STORE>
__host__ __device__ bool fac_run(const LineDesc<TS> &d, const FacGeom &g, const double *dBh, const double *dBt, TS *rec, int b0,
                        int b1, double (&G)[3][3]) {
    TS *recS = rec, *recF = rec + fac_part(g), *recH = rec + (size_t)2 * fac_part(g);
    const double bh2 = d.beta * d.inv_h * d.inv_h;
    const TS *__restrict__ al = d.alpha;
    const long long sp = d.sp;
    double F[3][3] = {}, H[3][3] = {};
    int c = b0 / g.mm, i = 0;
    for (int b = b0; b < b1; ++b) {
        const bool first = b == 0, last = b == g.nb - 1;
        const int cb = g.first + 3 * b;
        double sc[3], S[3][3], R[3][3];
#pragma unroll
        for (int m = 0; m < 3; ++m) sc[m] = (double)al[(cb + m) * sp] * bh2;
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int q = 0; q < 3; ++q) S[p][q] = fma_rn(-sc[p], mim_DG(q - p + 3), p == q ? 1.0 : 0.0);
        if (first)
            for (int p = 0; p < 3; ++p)
                for (int q = 0; q < 3; ++q) S[p][q] -= dBh[p * 3 + q];
        if (last)
            for (int p = 0; p < 3; ++p)
                for (int q = 0; q < 3; ++q) S[p][q] -= dBt[p * 3 + q];
        if (!first)  // S -= A G, A[p][k] = -s_p K_(3 + p - k) for k >= p
#pragma unroll
            for (int p = 0; p < 3; ++p)
#pragma unroll
                for (int k = p; k < 3; ++k) {
                    const double ak = mul_rn(sc[p], mim_DG(k - p));
#pragma unroll
                    for (int q = 0; q < 3; ++q) S[p][q] = fma_rn(ak, G[k][q], S[p][q]);
                }
        const double det = S[0][0] * (S[1][1] * S[2][2] - S[1][2] * S[2][1]) - S[0][1] * (S[1][0] * S[2][2] - S[1][2] * S[2][0]) +
                           S[0][2] * (S[1][0] * S[2][1] - S[1][1] * S[2][0]);
        if (!fac_pivot_ok(det)) return false;
        mat_inv<double, 3>(S, R);
#pragma unroll
        for (int q = 0; q < 3; ++q) {  // G = R C, C[k][q] = -s_k K_(3 + q - k) for q <= k
            double t[3] = {0.0, 0.0, 0.0};
#pragma unroll
            for (int k = q; k < 3; ++k) {
                const double ck = -mul_rn(sc[k], mim_DG(q - k + 6));
#pragma unroll
                for (int p = 0; p < 3; ++p) t[p] = fma_rn(R[p][k], ck, t[p]);
            }
#pragma unroll
            for (int p = 0; p < 3; ++p) G[p][q] = last ? 0.0 : t[p];
        }
        if constexpr (STORE) {
            double E[3][3];  // -R A
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                double t[3] = {0.0, 0.0, 0.0};
#pragma unroll
                for (int k = 0; k <= q; ++k) {
                    const double ak = mul_rn(sc[k], mim_DG(q - k));
#pragma unroll
                    for (int p = 0; p < 3; ++p) t[p] = fma_rn(R[p][k], ak, t[p]);
                }
#pragma unroll
                for (int p = 0; p < 3; ++p) E[p][q] = first ? 0.0 : t[p];
            }
            if (i == 0) {
                for (int p = 0; p < 3; ++p)
                    for (int q = 0; q < 3; ++q) {
                        recS[(size_t)c * 9 + p * 3 + q] = (TS)S[p][q];
                        F[p][q] = E[p][q];
                        H[p][q] = -G[p][q];
                    }
            } else {
                double f[3][3], h[3][3];
#pragma unroll
                for (int p = 0; p < 3; ++p)
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        f[p][q] = fma_rn(E[p][2], F[2][q], fma_rn(E[p][1], F[1][q], mul_rn(E[p][0], F[0][q])));
                        h[p][q] = -fma_rn(H[p][2], G[2][q], fma_rn(H[p][1], G[1][q], mul_rn(H[p][0], G[0][q])));
                    }
#pragma unroll
                for (int p = 0; p < 3; ++p)
#pragma unroll
                    for (int q = 0; q < 3; ++q) { F[p][q] = f[p][q]; H[p][q] = h[p][q]; }
            }
            if (++i == g.mm) {
                for (int p = 0; p < 3; ++p)
                    for (int q = 0; q < 3; ++q) {
                        recF[(size_t)c * 9 + p * 3 + q] = (TS)F[p][q];
                        recH[(size_t)c * 9 + p * 3 + q] = (TS)H[p][q];
                    }
                i = 0;
                ++c;
            }
        }
    }
    return true;
}

__host__ __device__ __forceinline__ float fac_abs(float x) { return x < 0.f ? -x : x; }
__host__ __device__ __forceinline__ double fac_abs(double x) { return x < 0.0 ? -x : x; }

// Reach of the windowed scans over the windows that start at the chunks [e0, e1) (see the header): the
// largest number of consecutive stored transfers (forward: F_e F_{e-1} ..., backward: H_s H_{s+1} ...)
// whose product first has infinity norm at most tau, or that reaches the end of the line; at most
// kFacMaxReach + 1 (which selects the full scan).
// A window's products are formed in FP32 with an entrywise bound on what its roundings have done, and again in FP64 where
// the bound leaves open on which side of tau a norm lies (the FP64 pipe is what the records wait for), so that the reach
// is FP64's.  The bound: with |P^ - P| <= E, the product P^ M^ of M^ = M (1 + 2^-24) as BS products and sums differs from P M
// by at most (E + (BS + 1) 2^-24 |P^|) |M|; 2^-21 in its place leaves room for FP64's roundings, 1e-36 for what FP32
// flushes, and 1 % and 2^-20 of the norm for the roundings of the bound and the norm themselves.  (Entrywise, because the
// rows of a CFD transfer differ in size: bounds by norms left so much open that most windows ran again.  1023 CFD lines of
// 1024 cells: 269 us for their records, 364 with such bounds, 367 in FP64 throughout, 267 without a bound.)
template <typename TS, int BS, typename R>
__host__ __device__ int fac_window(const TS *maps, int tact, double tau, bool forward, int first, bool &unsure) {
    constexpr int B2 = BS * BS;
    constexpr bool kBound = sizeof(R) == 4;
    R P[BS][BS], E[BS][BS];
#pragma unroll
    for (int p = 0; p < BS; ++p)
#pragma unroll
        for (int q = 0; q < BS; ++q) { P[p][q] = p == q ? R(1) : R(0); E[p][q] = R(0); }
    unsure = false;
    for (int r = 0;;) {
        const int k = forward ? first - r : first + r;
        R M[BS][BS], T1[BS][BS], E1[BS][BS], nrm = R(0), err = R(0);
#pragma unroll
        for (int p = 0; p < BS; ++p)
#pragma unroll
            for (int q = 0; q < BS; ++q) M[p][q] = (R)maps[(size_t)k * B2 + p * BS + q];
#pragma unroll
        for (int p = 0; p < BS; ++p) {
            R rs = R(0), es = R(0);
#pragma unroll
            for (int q = 0; q < BS; ++q) {
                R t = R(0), b = R(1e-36);
#pragma unroll
                for (int m = 0; m < BS; ++m) {
                    t += P[p][m] * M[m][q];
                    if (kBound) b += (E[p][m] + R(0x1p-21) * fac_abs(P[p][m])) * fac_abs(M[m][q]);
                }
                T1[p][q] = t;
                E1[p][q] = b;
                rs += fac_abs(t);
                es += b;
            }
            nrm = rs > nrm ? rs : nrm;
            err = es > err ? es : err;
        }
#pragma unroll
        for (int p = 0; p < BS; ++p)
#pragma unroll
            for (int q = 0; q < BS; ++q) { P[p][q] = T1[p][q]; E[p][q] = E1[p][q]; }
        ++r;
        if (kBound && !(fac_abs(nrm - (R)tau) > R(1.01) * err + R(0x1p-20) * nrm)) { unsure = true; return r; }
        const bool at_end = forward ? (k == 0) : (k == tact - 1);
        if (nrm <= (R)tau || at_end || r > kFacMaxReach) return r;
    }
}
template <typename TS, int BS>
__host__ __device__ int fac_reach(const TS *maps, int tact, double tau, bool forward, int e0, int e1) {
    int reach = 0;
    for (int e = e0; e < e1 && e < tact - 1 && reach <= kFacMaxReach; ++e) {
        const int first = forward ? e : e + 1;  // chunk whose transfer the window starts with
        bool unsure;
        int r = fac_window<TS, BS, float>(maps, tact, tau, forward, first, unsure);
        if (unsure) r = fac_window<TS, BS, double>(maps, tact, tau, forward, first, unsure);
        reach = r > reach ? r : reach;
    }
    return reach;
}

// The chunk records of the lines of one direction (all of N cells): segs threads per line, each the
// block LU of a run of whole chunks.  A run inside the line starts fac_warm blocks earlier from G = 0:
// the recursion forgets its start by the square of what the chunk transfers decay (on the seismic grids
// 0.4 a CFD block, 4e-26 over 64, and 0.01 an MFD block, 1e-32 over 16).  Whether it did is checked, not assumed: the G it
// reached at its first block must agree with the G of the run before (fac_same_start), else one thread
// does the line again from its head (weakly decaying lines, as with very large time steps).
constexpr int kFacRecThreads = 128;
__host__ __device__ inline int fac_warm(int method) { return method == kCFD ? 64 : 16; }
// Whether the run before ended where this one started, to two units in the last place of the largest entry: where alpha is
// constant the recursion's roundings settle in one of several neighbouring values, whichever way it came (asking for
// the same bits sent lines of layered media of 1024 cells the long way, 269 -> 2726 us for CFD's records and 324 -> 4936 for
// MFD's).  The error of the kept runs' records, against extended precision, is 0.66 to 1.08 times that of one run from the head,
// 0.99 on average, over media of four kinds and Courant numbers of 0.1 to 6; with 1e-15 it was up to 1.45 times.
__host__ __device__ inline bool fac_same_start(const double *start, const double *end, int n) {
    double size = 0.0;
    for (int i = 0; i < n; ++i) size = fmax(size, fabs(end[i]));
    bool same = true;
    for (int i = 0; i < n; ++i) same = same && fabs(start[i] - end[i]) <= 0x1p-51 * size;  // false for NaN
    return same;
}
template <typename TS, int BS>
__device__ void fac_records(const LineDesc<TS> &d, const FacGeom &g, const double *dB, int segs, int seg, bool mine,
                            double (*gs)[9], double (*ge)[9], int *bad, int *status) {
    const int c0 = (int)((long long)g.tact * seg / segs), c1 = (int)((long long)g.tact * (seg + 1) / segs);
    TS *rec = d.sep;
    const int t = threadIdx.x;
    bool ok = true;
    if (seg == 0) *bad = 0;
    if (mine) {
        double G[BS][BS] = {};
        const int b0 = c0 * g.mm;
        if (b0 > 0) ok = fac_run<TS, false>(d, g, dB, dB + 9, rec, max(0, b0 - fac_warm(d.method)), b0, G);
        for (int p = 0; p < BS; ++p)
            for (int q = 0; q < BS; ++q) gs[t][p * BS + q] = G[p][q];
        if (ok) ok = fac_run<TS, true>(d, g, dB, dB + 9, rec, b0, c1 * g.mm, G);
        for (int p = 0; p < BS; ++p)
            for (int q = 0; q < BS; ++q) ge[t][p * BS + q] = G[p][q];
    }
    __syncthreads();
    if (mine) {
        if (seg > 0) ok = ok && fac_same_start(gs[t], ge[t - 1], BS * BS);
        if (!ok) atomicExch(bad, 1);
    }
    __syncthreads();
    if (mine && seg == 0 && *bad) {
        double G[BS][BS] = {};
        if (!fac_run<TS, true>(d, g, dB, dB + 9, rec, 0, g.nb, G)) atomicExch(status, 1);
    }
    __syncthreads();  // the line's F and H are written (to global memory, by this block)
    if (!mine) return;
    const double tau = sizeof(TS) == 4 ? 0x1p-40 : 0x1p-70;
    const int rf = fac_reach<TS, BS>(rec + fac_part(g), g.tact, tau, true, c0, c1);
    const int rb = fac_reach<TS, BS>(rec + (size_t)2 * fac_part(g), g.tact, tau, false, c0, c1);
    gs[t][0] = rf;
    ge[t][0] = rb;
}

template <typename TS>
__global__ void __launch_bounds__(kFacRecThreads) fac_records_kernel(const LineDesc<TS> *__restrict__ descs, int nlines,
                                                                     int segs, const double *dB, int *status) {
    __shared__ double gs[kFacRecThreads][9], ge[kFacRecThreads][9];
    __shared__ int bad[kFacRecThreads];
    const int per = kFacRecThreads / segs, t = threadIdx.x;
    const int l = t / segs, seg = t % segs, line = blockIdx.x * per + l;
    const bool mine = line < nlines;
    const LineDesc<TS> &d = descs[mine ? line : 0];
    const FacGeom g = fac_geom(d.method, d.N);
    const double *db = dB + (size_t)(mine ? line : 0) * 18;
    if (d.method == kCFD) fac_records<TS, 2>(d, g, db, segs, seg, mine, gs, ge, bad + l, status);
    else fac_records<TS, 3>(d, g, db, segs, seg, mine, gs, ge, bad + l, status);
    __syncthreads();
    if (!mine || seg != 0) return;
    double rf = 0.0, rb = 0.0;
    for (int k = 0; k < segs; ++k) {
        rf = fmax(rf, gs[t + k][0]);
        rb = fmax(rb, ge[t + k][0]);
    }
    TS *info = d.sep + fac_info(g);
    info[0] = (TS)rf;
    info[1] = (TS)rb;
    info[2] = info[3] = (TS)0;
    atomicMax(status + 1, (int)fmax(rf, rb));
}

// ---------------------------------------------------------------------------------------
// Affine maps z -> m z + off and their segmented scans over the chunks of a line.
// ---------------------------------------------------------------------------------------
template <typename T, int BS>
struct Map {
    T m[BS][BS];
    T off[BS];
};
template <typename T, int BS>
__device__ __forceinline__ void map_id(Map<T, BS> &a) {
#pragma unroll
    for (int i = 0; i < BS; ++i) {
        a.off[i] = T(0);
#pragma unroll
        for (int j = 0; j < BS; ++j) a.m[i][j] = i == j ? T(1) : T(0);
    }
}
// a <- a o b  (b first, then a)
template <typename T, int BS>
__device__ __forceinline__ void map_after(Map<T, BS> &a, const Map<T, BS> &b) {
    Map<T, BS> r;
#pragma unroll
    for (int i = 0; i < BS; ++i) {
        T acc = a.off[i];
#pragma unroll
        for (int k = 0; k < BS; ++k) acc += a.m[i][k] * b.off[k];
        r.off[i] = acc;
#pragma unroll
        for (int j = 0; j < BS; ++j) {
            T s = T(0);
#pragma unroll
            for (int k = 0; k < BS; ++k) s += a.m[i][k] * b.m[k][j];
            r.m[i][j] = s;
        }
    }
    a = r;
}
template <typename T, int BS>
__device__ __forceinline__ void map_shfl(Map<T, BS> &dst, const Map<T, BS> &src, int delta, bool up, int width) {
#pragma unroll
    for (int i = 0; i < BS; ++i) {
#pragma unroll
        for (int j = 0; j < BS; ++j)
            dst.m[i][j] = up ? __shfl_up_sync(0xffffffffu, src.m[i][j], delta, width)
                             : __shfl_down_sync(0xffffffffu, src.m[i][j], delta, width);
        dst.off[i] = up ? __shfl_up_sync(0xffffffffu, src.off[i], delta, width)
                        : __shfl_down_sync(0xffffffffu, src.off[i], delta, width);
    }
}

// Barrier of the compute warps of a CTA of NT threads (named barrier 1; the staging warp does not take
// part).
template <int NT>
__device__ __forceinline__ void workers_sync() {
    asm volatile("bar.sync 1, %0;" ::"r"(NT - 32) : "memory");
}

// Scan buffers of a CTA: warp aggregates and warp prefixes.
template <typename T, int BS>
struct ScanSmem {
    Map<T, BS> agg[kFacThreads / 32];
    T pre[kFacThreads / 32][BS];
};

// Exclusive scan over the Tl chunk-threads of each line (lines occupy aligned groups of Tl
// consecutive threads; threads past the last whole line of the CTA take part in the warp
// shuffles only).  forward: z(c) = (a_{c-1} o ... o a_0)(0), the value entering chunk c;
// backward: z(c) = (a_{c+1} o ... o a_{Tl-1})(0), the value after chunk c.  Every thread of
// the CTA must call it with the same Tl.
template <typename T, int BS, int NT>
__device__ __forceinline__ void seg_scan(Map<T, BS> a, bool forward, int Tl, T (&z)[BS], ScanSmem<T, BS> &sm) {
    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const int width = Tl < 32 ? Tl : 32;
    const int pos = forward ? (lane % width) : (width - 1 - lane % width);
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
        if (s >= width) break;
        Map<T, BS> o;
        map_shfl<T, BS>(o, a, s, forward, width);
        if (pos >= s) map_after<T, BS>(a, o);
    }
    Map<T, BS> ex;
    map_shfl<T, BS>(ex, a, 1, forward, width);
    if (pos == 0) map_id<T, BS>(ex);
    if (Tl <= 32) {
#pragma unroll
        for (int i = 0; i < BS; ++i) z[i] = ex.off[i];
        return;
    }
    const int nw = Tl >> 5;          // warps per line
    const int wl = warp % nw;        // warp index within its line
    const bool whole = (tid / Tl) < ((NT - 32) / Tl);  // inside a whole line of the CTA
    if (pos == 31) sm.agg[warp] = a;  // the warp's full composition
    workers_sync<NT>();
    if (whole && wl == 0 && lane == 0) {
        T p[BS];
#pragma unroll
        for (int i = 0; i < BS; ++i) p[i] = T(0);
        for (int k = 0; k < nw; ++k) {
            const int w = warp + (forward ? k : nw - 1 - k);
#pragma unroll
            for (int i = 0; i < BS; ++i) sm.pre[w][i] = p[i];
            const Map<T, BS> &ag = sm.agg[w];
            T q[BS];
#pragma unroll
            for (int i = 0; i < BS; ++i) {
                T acc = ag.off[i];
#pragma unroll
                for (int k2 = 0; k2 < BS; ++k2) acc += ag.m[i][k2] * p[k2];
                q[i] = acc;
            }
#pragma unroll
            for (int i = 0; i < BS; ++i) p[i] = q[i];
        }
    }
    workers_sync<NT>();
#pragma unroll
    for (int i = 0; i < BS; ++i) {
        T acc = ex.off[i];
#pragma unroll
        for (int k = 0; k < BS; ++k) acc += ex.m[i][k] * sm.pre[warp][k];
        z[i] = acc;
    }
}

// Block inverse of the line kernel.  CFD in FP64 divides: with fac_rcp a step's error was no smaller (v and w 0.03 %
// larger) for 2 % of its time (512 x 512 cells: 108 us, 106 with it).
__device__ __forceinline__ float fac_block_rcp(float x) { return fac_rcp(x); }
__device__ __forceinline__ double fac_block_rcp(double x) { return 1.0 / x; }
template <typename T, int BS>
__device__ __forceinline__ void fac_inv(const T (&S)[BS][BS], T (&R)[BS][BS]) {
    if constexpr (BS == 2) {
        const T id = fac_block_rcp(S[0][0] * S[1][1] - S[0][1] * S[1][0]);
        R[0][0] = S[1][1] * id; R[0][1] = -S[0][1] * id;
        R[1][0] = -S[1][0] * id; R[1][1] = S[0][0] * id;
    } else {
        const T c00 = S[1][1] * S[2][2] - S[1][2] * S[2][1];
        const T c01 = S[1][2] * S[2][0] - S[1][0] * S[2][2];
        const T c02 = S[1][0] * S[2][1] - S[1][1] * S[2][0];
        const T id = fac_block_rcp(S[0][0] * c00 + S[0][1] * c01 + S[0][2] * c02);
        R[0][0] = c00 * id;
        R[0][1] = (S[0][2] * S[2][1] - S[0][1] * S[2][2]) * id;
        R[0][2] = (S[0][1] * S[1][2] - S[0][2] * S[1][1]) * id;
        R[1][0] = c01 * id;
        R[1][1] = (S[0][0] * S[2][2] - S[0][2] * S[2][0]) * id;
        R[1][2] = (S[0][2] * S[1][0] - S[0][0] * S[1][2]) * id;
        R[2][0] = c02 * id;
        R[2][1] = (S[0][1] * S[2][0] - S[0][0] * S[2][1]) * id;
        R[2][2] = (S[0][0] * S[1][1] - S[0][1] * S[1][0]) * id;
    }
}

// ---------------------------------------------------------------------------------------
// Bulk asynchronous copies (global -> shared) completing on an mbarrier.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_addr(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned long long *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_to_smem(void *dst, const void *src, unsigned bytes, unsigned long long *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long *bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Waits for the phase with the given parity; gives up after a bounded number of polls
// (each poll may suspend the thread for a short hardware-defined time).
__device__ __forceinline__ bool mbar_wait(unsigned long long *bar, unsigned parity, int polls = 1 << 22) {
    for (int i = 0; i < polls; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

__host__ __device__ inline unsigned round16(unsigned b) { return (b + 15u) & ~15u; }

// Bulk copies (shared -> global) of the staged outputs of a solved group, issued by the lanes
// of the staging warp once the compute warps have released the stage (lane k takes lines k,
// k + 32, ...); each line's pressure output (in place of its pressure line) and v' (in place
// of alpha).  Lines shorter than a warp were stored directly by the compute warps.  Returns
// once this lane's copies have read the stage.
template <typename T>
__device__ void fac_store_outputs(const unsigned char *stage, int lane) {
    const FacGroup &gr = *(const FacGroup *)stage;
    if (gr.T < 32) return;
    const LineDesc<T> *descs = (const LineDesc<T> *)(stage + kFacGroupBytes);
    const T *base = (const T *)(stage + fac_head_bytes(gr.nl));
    // stored spans [sp0, sp1) and [sv0, sv1): 4-element-aligned starts, lengths rounded up to
    // 16 bytes only at the line's end (inside the padded line)
    const unsigned pbytes = round16((unsigned)(gr.sp1 - gr.sp0) * (unsigned)sizeof(T));
    const unsigned vbytes = round16((unsigned)(gr.sv1 - gr.sv0) * (unsigned)sizeof(T));
    for (int l = lane; l < gr.nl; l += 32) {
        const T *sp = base + (size_t)l * gr.ls - gr.lo;  // staged element k at sp[k]
        if (pbytes)
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(descs[l].po + gr.sp0),
                         "r"(smem_addr(sp + gr.sp0)), "r"(pbytes)
                         : "memory");
        if (vbytes)
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(descs[l].vo + gr.sv0),
                         "r"(smem_addr(sp + 2 * gr.lp + gr.sv0)), "r"(vbytes)
                         : "memory");
    }
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

// The staging warp: stage one line group (descriptors, then per line the pressure, velocity
// and alpha lines and the record) into shared memory.  Lane 0 announces the group's bytes on the
// stage's "full" barrier (its only arrival) and copies the header and the descriptors; lane k
// issues the copies of lines k, k + 32, ..., whose addresses follow from the group's header alone.
// A sub-line of a split line stages its span of the three lines and, of the record, its chunks'
// S, F and H parts, the end tables it holds and the reach.  Every source starts on a 16-byte
// boundary (padded leading dimensions; spans start at multiples of four elements; record parts
// are padded to four elements and sub-line ranges start at multiples of four chunks) and the
// copies, rounded up to 16 bytes, stay inside the padded line or the record.
template <typename T, int BS, bool SPLIT>
__device__ void fac_issue(const LineDesc<T> *__restrict__ descs, const FacGroup *gp, unsigned char *stage,
                          unsigned long long *bar, int lane, int q) {
    const FacGroup &gr = *gp;
    const int Lp = gr.lp, lo = SPLIT ? gr.lo : 0;
    const unsigned bp = round16((unsigned)gr.pn * (unsigned)sizeof(T));
    const unsigned bv = round16((unsigned)gr.vn * (unsigned)sizeof(T));
    const unsigned br = (unsigned)(gr.info + 4) * (unsigned)sizeof(T);  // the staged record
    const unsigned bd = (unsigned)(gr.nl * kDescBytes);
    const unsigned bg = (unsigned)kFacGroupBytes;
    if (lane == 0) {
        mbar_expect_tx(bar, bg + bd + (unsigned)gr.nl * (2 * bp + bv + br));
        bulk_to_smem(stage, gp, bg, bar);
        bulk_to_smem(stage + kFacGroupBytes, descs + gr.first, bd, bar);
    }
    __syncwarp();  // the group's bytes are announced before any line copy is issued
    T *base = (T *)(stage + fac_head_bytes(gr.nl));
    const T *gp_ = (const T *)gr.gp, *gv_ = (const T *)gr.gv[q], *ga_ = (const T *)gr.ga, *gs_ = (const T *)gr.gs;
    for (int l = lane; l < gr.nl; l += 32) {
        T *ln = base + (size_t)l * gr.ls;
        const T *sep = gs_ + (size_t)l * gr.dr;
        bulk_to_smem(ln, gp_ + (size_t)l * gr.dp + lo, bp, bar);
        bulk_to_smem(ln + Lp, gv_ + (size_t)l * gr.dv + lo, bv, bar);
        bulk_to_smem(ln + 2 * Lp, ga_ + (size_t)l * gr.dp + lo, bp, bar);
        if constexpr (!SPLIT) {
            bulk_to_smem(ln + 3 * Lp, sep, br, bar);
        } else {
            const FacGeom g = fac_geom(BS == 2 ? kCFD : kMFD, gr.N);
            const int pg = fac_part(g), es = fac_e_stride(g);
            const size_t cs = (size_t)gr.c0 * (BS * BS);
            const unsigned bpart = (unsigned)gr.part * (unsigned)sizeof(T);
            const unsigned be = (unsigned)es * (unsigned)sizeof(T);
            T *rec = ln + 3 * Lp;
            const T *src = sep;
            bulk_to_smem(rec, src + cs, bpart, bar);
            bulk_to_smem(rec + gr.part, src + pg + cs, bpart, bar);
            bulk_to_smem(rec + 2 * gr.part, src + 2 * pg + cs, bpart, bar);
            if (gr.eh >= 0) bulk_to_smem(rec + gr.eh, src + 3 * pg, be, bar);
            if (gr.et >= 0) bulk_to_smem(rec + gr.et, src + 3 * pg + es, be, bar);
            bulk_to_smem(rec + gr.info, src + 3 * pg + 2 * es, 4u * (unsigned)sizeof(T), bar);
        }
    }
}

// W consecutive shared-memory elements into registers (the chunks' odd stride spreads the lanes
// over the banks).
template <typename T, int W>
__device__ __forceinline__ void load_win(const T *src, T (&w)[W]) {
#pragma unroll
    for (int k = 0; k < W; ++k) w[k] = src[k];
}

// BS x BS block from shared memory (16-byte load for a 2x2 FP32 block: records are 16-byte
// aligned and 2x2 blocks lie on 16-byte boundaries).
template <typename T, int BS>
__device__ __forceinline__ void load_blk(const T *src, T (&M)[BS][BS]) {
    if constexpr (sizeof(T) == 4 && BS == 2) {
        const float4 q = *reinterpret_cast<const float4 *>(src);
        M[0][0] = q.x; M[0][1] = q.y; M[1][0] = q.z; M[1][1] = q.w;
    } else {
#pragma unroll
        for (int p = 0; p < BS; ++p)
#pragma unroll
            for (int q = 0; q < BS; ++q) M[p][q] = src[p * BS + q];
    }
}

// Windowed scan value of chunk c (see the header): forward, the value entering c from the
// `reach` chunks before it, z <- F_k z + o_k for k = max(0, c - reach) .. c-1; backward, the
// value after c from the chunks after it, z <- H_k z + o_k for k = min(tact-1, c + reach) ..
// c+1.  maps: the line's F or H blocks; off: the line's chunk offsets (BS per chunk).
template <typename T, int BS>
__device__ __forceinline__ void win_scan(bool forward, int c, int tact, int reach, const T *maps, const T *off,
                                         T (&z)[BS]) {
    const int k0 = forward ? max(0, c - reach) : min(tact - 1, c + reach);
    const int n = forward ? c - k0 : k0 - c;
    // the first map of the window would act on zero: its chunk's value starts the recurrence
#pragma unroll
    for (int p = 0; p < BS; ++p) z[p] = n > 0 ? off[k0 * BS + p] : T(0);
#pragma unroll 4
    for (int t = 1; t < n; ++t) {
        const int k = forward ? k0 + t : k0 - t;
        T M[BS][BS];
        load_blk<T, BS>(maps + k * BS * BS, M);
        T nz[BS];
#pragma unroll
        for (int p = 0; p < BS; ++p) {
            T acc = off[k * BS + p];
#pragma unroll
            for (int q = 0; q < BS; ++q) acc += M[p][q] * z[q];
            nz[p] = acc;
        }
#pragma unroll
        for (int p = 0; p < BS; ++p) z[p] = nz[p];
    }
}

// An MFD chunk in FP64, eliminated row by row as a band matrix.  Row k is 1 - s K_0 on the diagonal and -s K_d
// at distance d = 1..3 (s = alpha beta / h^2, K the 7-point operator); Crout form: L_d the eliminated lower bands, q
// = 1 / pivot, v_d the eliminated upper bands times q.  About 31 FP64 operations a cell for the factors and
// the substitutions, against about 55 for 3 x 3 block products and inverses: the FP64 pipe bounds the kernel (1001
// lines of 1001 cells: 200 -> 144 us together with the cheaper reciprocals and the 256-thread CTAs).
// FP32 keeps the block form: three approximate reciprocals a block instead of one doubled its error (100 x 100 cells,
// 25 steps: 1.3e-6 -> 3.4e-6 of the 64-bit result) for 1-3 %.
template <int MM>
struct MfdBand {
    static constexpr int NC = 3 * MM;
    double L1[NC], L2[NC], L3[NC], q[NC], v1[NC], v2[NC];  // the third upper band is L3 q
    // Factors, and the block value y that leaves the chunk if none enters it.  S: the Schur complement of the
    // chunk's first block; dB: the tail region's correction of its last block, or nullptr.
    __device__ __forceinline__ void factor(const double (&al)[NC], double bh2, const double (&S)[3][3], const double *dB,
                                           const double (&Y)[MM][3], double (&yend)[3]) {
        double v3[NC], z[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const double sc = al[k] * bh2;
            double di = 1.0 - sc * mim_DG(3);
            double lo1 = -sc * mim_DG(2), lo2 = -sc * mim_DG(1), up1 = lo1, up2 = lo2;
            L3[k] = -sc * mim_DG(0);
            if (k < 3) {  // in-block entries
                di = S[k][k];
                if (k >= 1) lo1 = S[k][k >= 1 ? k - 1 : 0];
                if (k == 2) lo2 = S[k][0];
                if (k <= 1) up1 = S[k][k <= 1 ? k + 1 : 2];
                if (k == 0) up2 = S[k][2];
            } else if (k >= NC - 3 && dB) {
                const int p = k - (NC - 3);
                di -= dB[p * 3 + p];
                if (p >= 1) lo1 -= dB[p * 3 + p - 1];
                if (p == 2) lo2 -= dB[p * 3];
                if (p <= 1) up1 -= dB[p * 3 + p + 1];
                if (p == 0) up2 -= dB[2];
            }
            double zz = Y[k / 3][k % 3];
            if (k >= 3) {
                lo2 -= L3[k] * v1[k - 3];
                lo1 -= L3[k] * v2[k - 3];
                di -= L3[k] * v3[k - 3];
                zz -= L3[k] * z[k - 3];
            }
            if (k >= 2) {
                L2[k] = lo2;
                lo1 -= lo2 * v1[k - 2];
                di -= lo2 * v2[k - 2];
                up1 -= lo2 * v3[k - 2];
                zz -= lo2 * z[k - 2];
            }
            if (k >= 1) {
                L1[k] = lo1;
                di -= lo1 * v1[k - 1];
                up1 -= lo1 * v2[k - 1];
                up2 -= lo1 * v3[k - 1];
                zz -= lo1 * z[k - 1];
            }
            q[k] = fac_rcp(di);
            v1[k] = up1 * q[k];
            v2[k] = up2 * q[k];
            v3[k] = L3[k] * q[k];
            z[k] = zz * q[k];
        }
        yend[2] = z[NC - 1];
        yend[1] = z[NC - 2] - v1[NC - 2] * z[NC - 1];
        yend[0] = z[NC - 3] - v1[NC - 3] * yend[1] - v2[NC - 3] * z[NC - 1];
    }
    // Y: r -> the true forward values, from the block value yin that enters; xfirst: x of the first block if
    // nothing follows the chunk.
    __device__ __forceinline__ void forward(const double (&al)[NC], double bh2, const double (&yin)[3], double (&Y)[MM][3],
                                            double (&xfirst)[3]) {
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const double sc = al[m] * bh2;
#pragma unroll
            for (int p = m; p < 3; ++p) Y[0][m] += sc * mim_DG(p - m) * yin[p];
        }
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            double a = Y[k / 3][k % 3];
            if (k >= 3) a -= L3[k] * Y[(k - 3) / 3][(k - 3) % 3];
            if (k >= 2) a -= L2[k] * Y[(k - 2) / 3][(k - 2) % 3];
            if (k >= 1) a -= L1[k] * Y[(k - 1) / 3][(k - 1) % 3];
            Y[k / 3][k % 3] = a * q[k];
            L3[k] *= q[k];  // from here on the third upper band
        }
        double x1 = 0.0, x2 = 0.0, x3 = 0.0;
#pragma unroll
        for (int k = NC - 1; k >= 0; --k) {
            const double x = Y[k / 3][k % 3] - L3[k] * x3 - v2[k] * x2 - v1[k] * x1;
            x3 = x2; x2 = x1; x1 = x;
        }
        xfirst[0] = x1; xfirst[1] = x2; xfirst[2] = x3;
    }
    // Y -> x, from the x that follows the chunk.
    __device__ __forceinline__ void backward(const double (&xin)[3], double (&Y)[MM][3]) {
        double x1 = xin[0], x2 = xin[1], x3 = xin[2];
#pragma unroll
        for (int k = NC - 1; k >= 0; --k) {
            const double x = Y[k / 3][k % 3] - L3[k] * x3 - v2[k] * x2 - v1[k] * x1;
            Y[k / 3][k % 3] = x;
            x3 = x2; x2 = x1; x1 = x;
        }
    }
};

// ---------------------------------------------------------------------------------------
// One line group from its staged inputs: nl lines of one simulation and direction, Tl
// threads per line; thread (l, c) = (tid / Tl, tid % Tl) owns middle blocks [c MM, c MM + MM).
// ---------------------------------------------------------------------------------------
template <typename T, int BS, int MM, bool SPLIT, int NT>
__device__ __forceinline__ void fac_group(unsigned char *stage_raw, int natural, ScanSmem<T, BS> &ssm,
                                          T *offf, T *offb) {
    static_assert(MM >= 2, "chunks of at least two blocks");
    using E = FacEnd<BS>;
    constexpr int W = E::W;
    static_assert(2 * W <= 32, "a window row fits one warp");
    constexpr int B2 = BS * BS;
    const int tid = threadIdx.x, lane = tid & 31;
    const FacGroup &gr = *(const FacGroup *)stage_raw;  // staged with the lines
    const LineDesc<T> *descs = (const LineDesc<T> *)(stage_raw + kFacGroupBytes);
    T *stage = (T *)(stage_raw + fac_head_bytes(gr.nl));
    const int N = gr.N, Tl = gr.T, tact = gr.tact;  // tact: chunks of the group's range
    const int Lp = gr.lp;
    const int l = Tl > 1 ? (int)__umulhi((unsigned)tid, gr.tdiv) : tid, c = tid - l * Tl;  // c: local chunk
    // a sub-line of a split line (SPLIT) covers the chunks c0 .. c0 + tact - 1 of its line
    const int cg = SPLIT ? gr.c0 + c : c;  // global chunk
    const int own = gr.own, ol0 = own & 511, ol1 = (own >> 9) & 511;
    const bool full_scan = (own & kFacOwnFull) != 0;
    const bool has_head = !SPLIT || (own & kFacOwnHead) != 0, has_tail = !SPLIT || (own & kFacOwnTail) != 0;
    const bool line_ok = l < gr.nl;
    const bool act = line_ok && c < tact;
    const bool owned = SPLIT ? act && c >= ol0 && c < ol1 : act;  // writes its outputs
    // an owned chunk at either end of a sub-line's owned span has outputs outside the
    // bulk-stored spans
    const bool edge = SPLIT && (c == ol0 || c == ol1 - 1);
    const int ll = line_ok ? l : 0;
    const LineDesc<T> &d = descs[ll];
    T *lb = stage + (size_t)ll * gr.ls;     // the line's staged block
    T *sPw = SPLIT ? lb - gr.lo : lb;       // staged element k of the pressure line at sPw[k]
    const T *sP = sPw;
    const T *sV = sP + Lp, *sA = sP + 2 * Lp, *sR = lb + 3 * Lp;
    const T *eH = sR + gr.eh, *eT = sR + gr.et;
    const int pl = gr.pl;
    constexpr int Z = E::Z;
    const T *sinfo = sR + gr.info;
    T *lofff = offf + (tid - c) * BS, *loffb = offb + (tid - c) * BS;  // this line's chunk offsets
    const T ih = sizeof(T) == 4 ? (T)gr.ihf : (T)gr.ih, beta = sizeof(T) == 4 ? (T)gr.betaf : (T)gr.beta;
    // segment of lanes that evaluates a line end: the whole warp for Tl >= 32, else the line
    const int S = Tl < 32 ? Tl : 32;
    const int ls = c & (S - 1);           // lane index within the segment (S a power of two)
    const int sbase = lane - ls;          // first lane of the segment
    const int wl = c >> 5;                // warp index within the line (Tl >= 32)
    const bool head_seg = has_head && (Tl < 32 || wl == 0);
    const bool tail_seg = has_tail && (Tl < 32 || wl == ((tact - 1) >> 5));
    const bool is_tail = act && has_tail && c == tact - 1;
    const int opT = pl + 1 - W, ovT = N + 1 - W;  // tail windows

    // ---- right-hand sides and the alpha window ----
    constexpr int NA = (BS == 2) ? MM + 2 : 3 * MM;
    T aw[NA];     // CFD: 3 alpha / h at nodes jb-1 .. jb+MM;  MFD: alpha at the chunk's cells
    T Y[MM][BS];  // r, then y, then x
    const int jb = gr.mid + cg * MM;      // CFD: first node of the chunk
    const int cb = gr.mid + 3 * cg * MM;  // MFD: first cell of the chunk
    if (act) {
        if constexpr (BS == 2) {
            const T c3 = T(3) * ih;
            T w[MM + 2];
            load_win<T, MM + 2>(sA + jb - 1, w);
#pragma unroll
            for (int k = 0; k < NA; ++k) aw[k] = c3 * w[k];
            load_win<T, MM + 2>(sV + jb - 1, w);
#pragma unroll
            for (int i = 0; i < MM; ++i) Y[i][0] = c3 * (w[i + 2] - w[i]);
            load_win<T, MM + 2>(sP + jb - 1, w);
#pragma unroll
            for (int i = 0; i < MM; ++i) Y[i][1] = c3 * (w[i + 2] - w[i]);
        } else {
#pragma unroll
            for (int k = 0; k < NA; ++k) aw[k] = sA[cb + k];
            T vw[3 * MM + 3];
#pragma unroll
            for (int k = 0; k < 3 * MM + 3; ++k) vw[k] = sV[cb - 2 + k];
            const T w0 = T(1.0 / 24.0), w1 = T(-9.0 / 8.0), w2 = T(9.0 / 8.0), w3 = T(-1.0 / 24.0);
#pragma unroll
            for (int i = 0; i < MM; ++i)
#pragma unroll
                for (int m = 0; m < 3; ++m) {
                    const int k = 3 * i + m;
                    const T dv = w0 * vw[k] + w1 * vw[k + 1] + w2 * vw[k + 2] + w3 * vw[k + 3];
                    Y[i][m] = sP[cb + k] - aw[k] * ih * dv;
                }
        }
    }

    // ---- head / tail corrections of the adjacent blocks' right-hand sides (KZ z) ----
    auto zval = [&](bool tail, int k) -> T {
        return k < W ? sP[(tail ? opT : 0) + k] : sV[(tail ? ovT : 0) + k - W];
    };
    // Window parts (first 2W terms) of the end-region rows HZ and DZ, known once the line is
    // staged: computed now by threads spread over the line and kept in the line's scratch, so
    // that at the end the end-region lanes add only the adjacent block's BS terms.
    // Row r < NR1 belongs to the head, r >= NR1 to the tail; within an end, HZ rows come first.
    constexpr int NR1 = E::HMAX + (BS == 3 ? E::HMAX + 2 : 0), NR = 2 * NR1;
    T *scr = lb + gr.scr;
    // Lines of at least three warps: the warps other than the head and tail warps compute the
    // rows after their local forward pass (below), while the end warps form KZ z.
    const bool scr_help = Tl >= 96;
    if (line_ok && !scr_help) {
        auto row_win = [&](int r) {
            const bool tail = r >= NR1;
            if (!(tail ? has_tail : has_head)) return;
            const int q = tail ? r - NR1 : r;
            const T *row = (tail ? eT : eH) + (q < E::HMAX ? E::HZ + q * Z : E::DZ + (q - E::HMAX) * Z);
            T a0 = T(0), a1 = T(0);
    #pragma unroll
            for (int k = 0; k < 2 * W; k += 2) {
                a0 += row[k] * zval(tail, k);
                a1 += row[k + 1] * zval(tail, k + 1);
            }
            scr[r] = a0 + a1;
        };
        const int stride = Tl >= NR ? Tl / NR : 1;
        if (stride > 1) {
            if (c % stride == 0 && c / stride < NR) row_win(c / stride);
        } else {
            for (int r = c; r < NR; r += Tl) row_win(r);
        }
    }
    auto seg_kz = [&](bool tail, T (&out)[BS]) {
        const T *kz = (tail ? eT : eH);
        if (S == 32) {  // one window term per lane (2W <= 32), then a warp sum
            const int k = ls;
            const bool has = k < 2 * W;
            const T *zp = k < W ? sP + (tail ? opT : 0) + k : sV + (tail ? ovT : 0) + (k - W);
            const T z = has ? *zp : T(0);
#pragma unroll
            for (int p = 0; p < BS; ++p) out[p] = has ? kz[p * 2 * W + k] * z : T(0);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int p = 0; p < BS; ++p) out[p] += __shfl_xor_sync(0xffffffffu, out[p], o);
            return;
        }
#pragma unroll
        for (int p = 0; p < BS; ++p) {
            T acc = T(0);
            for (int k = ls; k < 2 * W; k += S) acc += kz[p * 2 * W + k] * zval(tail, k);
            out[p] = acc;
        }
        for (int o = S >> 1; o > 0; o >>= 1)
#pragma unroll
            for (int p = 0; p < BS; ++p) out[p] += __shfl_xor_sync(0xffffffffu, out[p], o, S);
    };
    if (head_seg) {
        T kz[BS];
        seg_kz(false, kz);
        if (act && c == 0)
#pragma unroll
            for (int p = 0; p < BS; ++p) Y[0][p] += kz[p];
    }
    if (tail_seg) {
        T kz[BS];
        seg_kz(true, kz);
        if (is_tail)
#pragma unroll
            for (int p = 0; p < BS; ++p) Y[MM - 1][p] += kz[p];
    }

    // ---- block couplings from the alpha window ----
    // CFD: A_i = [[1, -tb], [-a_i, 1]], B = 4 I, C_i = [[1, tb], [a_{i+2}, 1]] with a = aw (3 alpha
    // / h at the nodes) and tb = 3 beta / h; its products below are written out, so that no unit
    // or zero entry costs an operation.  MFD: A_i (upper triangular), B_i and C_i (lower
    // triangular) hold the 7-point operator's bands scaled per cell; its products visit the
    // nonzero entries only (the compiler keeps a product with a literal zero).
    const T tb = T(3) * ih * beta;
    auto blockA = [&](int i, T (&A)[BS][BS]) {  // MFD
        const T bh2 = beta * ih * ih;
#pragma unroll
        for (int m = 0; m < BS; ++m) {
            const T sc = aw[3 * i + m] * bh2;
#pragma unroll
            for (int q = 0; q < BS; ++q) A[m][q] = (q >= m) ? -sc * (T)mim_DG(q - m) : T(0);
        }
    };
    auto blockB = [&](int i, T (&B)[BS][BS]) {  // MFD
        const T bh2 = beta * ih * ih;
#pragma unroll
        for (int m = 0; m < BS; ++m) {
            const T sc = aw[3 * i + m] * bh2;
#pragma unroll
            for (int q = 0; q < BS; ++q) B[m][q] = (q == m ? T(1) : T(0)) - sc * (T)mim_DG(q - m + 3);
        }
    };
    auto blockC = [&](int i, T (&C)[BS][BS]) {  // MFD
        const T bh2 = beta * ih * ih;
#pragma unroll
        for (int m = 0; m < BS; ++m) {
            const T sc = aw[3 * i + m] * bh2;
#pragma unroll
            for (int q = 0; q < BS; ++q) C[m][q] = (q <= m) ? -sc * (T)mim_DG(q - m + 6) : T(0);
        }
    };
    // out = A_i v
    auto mulA = [&](int i, const T (&v)[BS], T (&out)[BS]) {
        T r[BS];
        if constexpr (BS == 2) {
            r[0] = v[0] - tb * v[1];
            r[1] = v[1] - aw[i] * v[0];
        } else {
            T A[BS][BS];
            blockA(i, A);
#pragma unroll
            for (int p = 0; p < BS; ++p) {
                T acc = A[p][p] * v[p];
#pragma unroll
                for (int q = p + 1; q < BS; ++q) acc += A[p][q] * v[q];
                r[p] = acc;
            }
        }
#pragma unroll
        for (int p = 0; p < BS; ++p) out[p] = r[p];
    };
    // out = C_i v
    auto mulC = [&](int i, const T (&v)[BS], T (&out)[BS]) {
        T r[BS];
        if constexpr (BS == 2) {
            r[0] = v[0] + tb * v[1];
            r[1] = v[1] + aw[i + 2] * v[0];
        } else {
            T C[BS][BS];
            blockC(i, C);
#pragma unroll
            for (int p = 0; p < BS; ++p) {
                T acc = C[p][0] * v[0];
#pragma unroll
                for (int q = 1; q <= p; ++q) acc += C[p][q] * v[q];
                r[p] = acc;
            }
        }
#pragma unroll
        for (int p = 0; p < BS; ++p) out[p] = r[p];
    };
    // out = -Si t
    auto neg_si = [&](const T (&Si)[BS][BS], const T (&t)[BS], T (&out)[BS]) {
        T r[BS];
#pragma unroll
        for (int p = 0; p < BS; ++p) {
            T acc = Si[p][0] * t[0];
#pragma unroll
            for (int q = 1; q < BS; ++q) acc += Si[p][q] * t[q];
            r[p] = -acc;
        }
#pragma unroll
        for (int p = 0; p < BS; ++p) out[p] = r[p];
    };

    // ---- factorisation and local forward pass ----
    constexpr bool kBand = BS == 3 && sizeof(T) == 8;
    T Si[kBand ? 1 : MM][BS][BS];
    [[maybe_unused]] MfdBand<BS == 3 ? MM : 2> band;  // MFD in FP64
    T yend[BS], xfirst[BS];  // the chunk's y at its end if none enters it; x at its start if none follows
#pragma unroll
    for (int p = 0; p < BS; ++p) yend[p] = xfirst[p] = T(0);
    if constexpr (kBand) {
        if (act) {
            T S[BS][BS];
            load_blk<T, BS>(sR + c * B2, S);
            band.factor(aw, beta * ih * ih, S, is_tail ? eT + E::DB : nullptr, Y, yend);
        }
    } else if (act) {
        T G[BS][BS];
#pragma unroll
        for (int i = 0; i < MM; ++i) {
            T S[BS][BS];
            if (i == 0) {
                load_blk<T, BS>(sR + c * B2, S);
            } else {
                // S_i = B_i - A_i G_{i-1}
                if constexpr (BS == 2) {
                    S[0][0] = T(4) - G[0][0] + tb * G[1][0];
                    S[0][1] = tb * G[1][1] - G[0][1];
                    S[1][0] = aw[i] * G[0][0] - G[1][0];
                    S[1][1] = T(4) - G[1][1] + aw[i] * G[0][1];
                } else {
                    T A[BS][BS], B[BS][BS];
                    blockA(i, A);
                    blockB(i, B);
#pragma unroll
                    for (int p = 0; p < BS; ++p)
#pragma unroll
                        for (int q = 0; q < BS; ++q) {
                            T acc = B[p][q];
#pragma unroll
                            for (int k = p; k < BS; ++k) acc -= A[p][k] * G[k][q];
                            S[p][q] = acc;
                        }
                }
                if (i == MM - 1 && is_tail) {
#pragma unroll
                    for (int p = 0; p < BS; ++p)
#pragma unroll
                        for (int q = 0; q < BS; ++q) S[p][q] -= eT[E::DB + p * BS + q];
                }
            }
            fac_inv<T, BS>(S, Si[i]);
            // y_i = Si_i (r_i - A_i y_{i-1})
            T t[BS];
            if (i == 0) {
#pragma unroll
                for (int p = 0; p < BS; ++p) t[p] = Y[0][p];
            } else if constexpr (BS == 2) {
                t[0] = Y[i][0] - Y[i - 1][0] + tb * Y[i - 1][1];
                t[1] = Y[i][1] - Y[i - 1][1] + aw[i] * Y[i - 1][0];
            } else {
                T A[BS][BS];
                blockA(i, A);
#pragma unroll
                for (int p = 0; p < BS; ++p) {
                    T acc = Y[i][p];
#pragma unroll
                    for (int q = p; q < BS; ++q) acc -= A[p][q] * Y[i - 1][q];
                    t[p] = acc;
                }
            }
#pragma unroll
            for (int p = 0; p < BS; ++p) {
                T acc = Si[i][p][0] * t[0];
#pragma unroll
                for (int q = 1; q < BS; ++q) acc += Si[i][p][q] * t[q];
                Y[i][p] = acc;
            }
            if (i + 1 < MM) {  // G_i = Si_i C_i
                if constexpr (BS == 2) {
                    const T a2 = aw[i + 2];
                    G[0][0] = Si[i][0][0] + Si[i][0][1] * a2;
                    G[0][1] = Si[i][0][0] * tb + Si[i][0][1];
                    G[1][0] = Si[i][1][0] + Si[i][1][1] * a2;
                    G[1][1] = Si[i][1][0] * tb + Si[i][1][1];
                } else {
                    T C[BS][BS];
                    blockC(i, C);
#pragma unroll
                    for (int p = 0; p < BS; ++p)
#pragma unroll
                        for (int q = 0; q < BS; ++q) {
                            T acc = Si[i][p][q] * C[q][q];
#pragma unroll
                            for (int k = q + 1; k < BS; ++k) acc += Si[i][p][k] * C[k][q];
                            G[p][q] = acc;
                        }
                }
            }
        }
#pragma unroll
        for (int p = 0; p < BS; ++p) yend[p] = Y[MM - 1][p];
    }

    // ---- window parts of the end-region rows by the middle warps.  A line with five or more takes one
    // row per half-warp (one or two terms per lane, then a half-warp sum): one to three passes.  A
    // shorter line's two to four would make up to 18, which took 2300 of a 128-thread line's 9600
    // cycles: there two of them take one row per lane, head and tail, adding the terms in the half-warp's order ----
    if (scr_help && line_ok) {
        const int tw = (tact - 1) >> 5;  // the tail warp (tact > 64, so 2 <= tw)
        if (wl != 0 && wl != tw) {
            const int hi = wl - 1 - (wl > tw ? 1 : 0), nh = (Tl >> 5) - 2;
            if (nh < 5) {
                static_assert(NR1 <= 32, "an end's rows fit one warp");
                auto row_tree = [&](bool tail) {
                    if (!(tail ? has_tail : has_head) || lane >= NR1) return;
                    const T *row = (tail ? eT : eH) + (lane < E::HMAX ? E::HZ + lane * Z : E::DZ + (lane - E::HMAX) * Z);
                    T a[16];
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        a[k] = mul_rn(row[k], zval(tail, k));
                        if (k + 16 < 2 * W) a[k] = fma_rn(row[k + 16], zval(tail, k + 16), a[k]);
                    }
#pragma unroll
                    for (int o = 8; o > 0; o >>= 1)
#pragma unroll
                        for (int k = 0; k < o; ++k) a[k] += a[k + o];
                    scr[(tail ? NR1 : 0) + lane] = a[0];
                };
                if (hi == 0) row_tree(false);
                if (hi == (nh > 1 ? 1 : 0)) row_tree(true);
            } else {
                const int half = lane >> 4, k = lane & 15;
                for (int r0 = 2 * hi; r0 < NR; r0 += 2 * nh) {  // warp-uniform trip count
                    const int r = r0 + half;
                    const bool tail = r >= NR1;
                    const int q = tail ? r - NR1 : r;
                    T a = T(0);
                    const bool here = r < NR && (tail ? has_tail : has_head);
                    if (here) {
                        const T *row = (tail ? eT : eH) + (q < E::HMAX ? E::HZ + q * Z : E::DZ + (q - E::HMAX) * Z);
                        a = row[k] * zval(tail, k);
                        if (k + 16 < 2 * W) a += row[k + 16] * zval(tail, k + 16);
                    }
#pragma unroll
                    for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
                    if (k == 0 && here) scr[r] = a;
                }
            }
        }
    }

    // ---- forward scan: the true y entering the chunk; correction ----
    T yin[BS];
    if (full_scan) {
        Map<T, BS> mp;
        if (act) {
            load_blk<T, BS>(sR + gr.part + c * B2, mp.m);
#pragma unroll
            for (int p = 0; p < BS; ++p) mp.off[p] = yend[p];
        } else {
            map_id<T, BS>(mp);
        }
        seg_scan<T, BS, NT>(mp, true, Tl, yin, ssm);
    } else {
        if (offb == offf) workers_sync<NT>();  // one offset buffer: the group before has read its values
        if (act)
#pragma unroll
            for (int p = 0; p < BS; ++p) lofff[c * BS + p] = yend[p];
        workers_sync<NT>();
        if (act) win_scan<T, BS>(true, c, tact, (int)sinfo[0], sR + gr.part, lofff, yin);
    }
    if constexpr (kBand) {
        if (act) band.forward(aw, beta * ih * ih, yin, Y, xfirst);
    } else if (act) {
        T dl[BS];
#pragma unroll
        for (int p = 0; p < BS; ++p) dl[p] = yin[p];
#pragma unroll
        for (int i = 0; i < MM; ++i) {  // d_i = -Si_i A_i d_{i-1}
            T t[BS];
            mulA(i, dl, t);
            neg_si(Si[i], t, dl);
#pragma unroll
            for (int p = 0; p < BS; ++p) Y[i][p] += dl[p];
        }
        // local backward pass (x = 0 after the chunk): x_i = y_i - Si_i (C_i x_{i+1})
#pragma unroll
        for (int i = MM - 2; i >= 0; --i) {
            T t[BS], u[BS];
            mulC(i, Y[i + 1], t);
            neg_si(Si[i], t, u);
#pragma unroll
            for (int p = 0; p < BS; ++p) Y[i][p] += u[p];
        }
#pragma unroll
        for (int p = 0; p < BS; ++p) xfirst[p] = Y[0][p];
    }

    // ---- backward scan: the true x after the chunk; correction ----
    T xin[BS];
    if (full_scan) {
        Map<T, BS> mp;
        if (act) {
            load_blk<T, BS>(sR + 2 * gr.part + c * B2, mp.m);
#pragma unroll
            for (int p = 0; p < BS; ++p) mp.off[p] = xfirst[p];
        } else {
            map_id<T, BS>(mp);
        }
        seg_scan<T, BS, NT>(mp, false, Tl, xin, ssm);
    } else {
        if (offb == offf) workers_sync<NT>();  // one offset buffer: the forward reads are done
        if (act)
#pragma unroll
            for (int p = 0; p < BS; ++p) loffb[c * BS + p] = xfirst[p];
        workers_sync<NT>();
        if (act) win_scan<T, BS>(false, c, tact, (int)sinfo[1], sR + 2 * gr.part, loffb, xin);
    }
    if constexpr (kBand) {
        if (act) band.backward(xin, Y);
    } else if (act) {
        T ep[BS];
#pragma unroll
        for (int p = 0; p < BS; ++p) ep[p] = xin[p];
#pragma unroll
        for (int i = MM - 1; i >= 0; --i) {  // e_i = -Si_i C_i e_{i+1}
            T t[BS];
            mulC(i, ep, t);
            neg_si(Si[i], t, ep);
#pragma unroll
            for (int p = 0; p < BS; ++p) Y[i][p] += ep[p];
        }
    }

    // ---- outputs: C = 2 u* - a (+ source), v' = 2 v* - v, optionally natural u, w ----
    T *__restrict__ gpo = d.po;
    T *__restrict__ gvo = d.vo;
    T *__restrict__ uo = natural ? d.u_out : nullptr;
    T *__restrict__ wo = natural ? d.w_out : nullptr;
    const long long spo = d.spo, svo = d.svo, snp = d.snp, snv = d.snv;
    const int src_k = d.src_k;
    // Lines of at least a warp stage their outputs in shared memory and leave with one bulk
    // copy per line and array: the pressure output in place of the pressure line, v' in
    // place of alpha.  Both are dead once the solve is done, and every thread reads them only
    // at the points it writes, before writing there.  Shorter lines store directly.
    const bool stage_v = Tl >= 32;
    T *sOut = sPw + 2 * Lp;
    // source term dt/2 f(t_{m+1}) added by the thread that wrote pressure point src_k
    // staged in shared memory inside the bulk-stored spans, stored directly outside them
    const int sp0 = gr.sp0, sp1 = gr.sp1, sv0 = gr.sv0, sv1 = gr.sv1;
    auto staged_p = [&](int k) { return SPLIT ? stage_v && k >= sp0 && k < sp1 : stage_v; };
    auto staged_v = [&](int j) { return SPLIT ? stage_v && j >= sv0 && j < sv1 : stage_v; };
    auto add_source = [&]() {
        const long long m = *d.clock;
        const T s = (T)(d.src_scale * ricker(d.src_amp, d.src_f0, d.src_tdelay, (double)(m + 1) * d.dt));
        if (staged_p(src_k)) sPw[src_k] += s; else gpo[src_k * spo] = gpo[src_k * spo] + s;
        if (d.advance_clock) *d.clock = m + 1;
    };
    // the fourth-order staggered difference of four consecutive values, up to the factor 1/h
    auto d4 = [](T a, T b, T c, T d) {
        return fma_rn(T(-1.0 / 24.0), d, fma_rn(T(9.0 / 8.0), c, fma_rn(T(-9.0 / 8.0), b, T(1.0 / 24.0) * a)));
    };
    auto out_p = [&](int k, T val_out, T val_nat) {
        if (staged_p(k)) sPw[k] = val_out; else gpo[k * spo] = val_out;
        if (uo) uo[k * snp] = val_nat;
    };
    // v' = v - 2 c g and the natural w = v - c g, with g the velocity's derivative term and c its
    // factor (beta for CFD, beta/h for MFD).  The carried value is formed exactly as on the
    // staged-only paths below, so that writing natural outputs never changes the trajectory.
    auto out_v = [&](int j, T vin, T cf, T g) {
        const T val = fma_rn(-(T(2) * cf), g, vin);
        if (staged_v(j)) sOut[j] = val; else gvo[j * svo] = val;
        if (wo) wo[j * snv] = fma_rn(-cf, g, vin);
    };
    if (owned) {
        if constexpr (BS == 2) {
            // alpha at the chunk's nodes is aw / (3/h); p and v at the chunk's nodes
            const T inv_c3 = T(1) / (T(3) * ih);
            T wp[MM], wv[MM];
            load_win<T, MM>(sP + jb, wp);
            load_win<T, MM>(sV + jb, wv);
            if (stage_v && !uo && !wo && !edge) {
#pragma unroll
                for (int i = 0; i < MM; ++i) {
                    const T ae = aw[i + 1] * inv_c3 * Y[i][0];
                    sPw[jb + i] = wp[i] - T(2) * ae;
                    sOut[jb + i] = fma_rn(-(T(2) * beta), Y[i][1], wv[i]);
                }
            } else {
#pragma unroll
                for (int i = 0; i < MM; ++i) {
                    const T ae = aw[i + 1] * inv_c3 * Y[i][0];
                    out_p(jb + i, wp[i] - T(2) * ae, wp[i] - ae);
                    out_v(jb + i, wv[i], beta, Y[i][1]);
                }
            }
            if (src_k >= jb && src_k < jb + MM) add_source();
        } else {
            const T bi = beta * ih;
            if (stage_v && !uo && !wo && !edge) {
                // staged outputs only: no per-point branches; the velocities after the last
                // block of the tail chunk belong to the tail region
                const T b2 = T(2) * bi;
#pragma unroll
                for (int i = 0; i < MM; ++i) {
                    const int q0 = cb + 3 * i;
#pragma unroll
                    for (int m = 0; m < 3; ++m) sPw[q0 + m] = T(2) * Y[i][m] - sP[q0 + m];
                    const T xn0 = i + 1 < MM ? Y[i + 1 < MM ? i + 1 : i][0] : xin[0];
                    const T xn1 = i + 1 < MM ? Y[i + 1 < MM ? i + 1 : i][1] : xin[1];
                    const T xn2 = i + 1 < MM ? Y[i + 1 < MM ? i + 1 : i][2] : xin[2];
                    const T d1 = d4(Y[i][0], Y[i][1], Y[i][2], xn0);
                    const T d2 = d4(Y[i][1], Y[i][2], xn0, xn1);
                    const T d3 = d4(Y[i][2], xn0, xn1, xn2);
                    if (i + 1 < MM || !is_tail) {
                        sOut[q0 + 1] = fma_rn(-b2, d1, sV[q0 + 1]);
                        sOut[q0 + 2] = fma_rn(-b2, d2, sV[q0 + 2]);
                        sOut[q0 + 3] = fma_rn(-b2, d3, sV[q0 + 3]);
                    }
                }
                if (src_k >= cb && src_k < cb + 3 * MM) add_source();
            } else {
#pragma unroll
            for (int i = 0; i < MM; ++i) {
                const int q0 = cb + 3 * i;
#pragma unroll
                for (int m = 0; m < 3; ++m) out_p(q0 + m, T(2) * Y[i][m] - sP[q0 + m], Y[i][m]);
                // x of the next block (the next chunk's first block after the last one)
                const int in = i + 1 < MM ? i + 1 : i;
                const T xn0 = i + 1 < MM ? Y[in][0] : xin[0];
                const T xn1 = i + 1 < MM ? Y[in][1] : xin[1];
                const T xn2 = i + 1 < MM ? Y[in][2] : xin[2];
                if (!(i == MM - 1 && is_tail)) {
                    out_v(q0 + 1, sV[q0 + 1], bi, d4(Y[i][0], Y[i][1], Y[i][2], xn0));
                    out_v(q0 + 2, sV[q0 + 2], bi, d4(Y[i][1], Y[i][2], xn0, xn1));
                    out_v(q0 + 3, sV[q0 + 3], bi, d4(Y[i][2], xn0, xn1, xn2));
                }
            }
            if (src_k >= cb && src_k < cb + 3 * MM) add_source();
            }
        }
    }

    // ---- head and tail regions, evaluated by their segments ----
    auto seg_end = [&](bool tail) {
        const T *et = tail ? eT : eH;
        const int src_lane = sbase + ((tail ? tact - 1 : 0) & (S - 1));
        T xJ[BS];
#pragma unroll
        for (int b = 0; b < BS; ++b) xJ[b] = __shfl_sync(0xffffffffu, tail ? Y[MM - 1][b] : Y[0][b], src_lane);
        if (!line_ok) return;
        const int m = tail ? gr.tu : gr.hu;
        const T *pscr = scr + (tail ? NR1 : 0);
        // row = [window part (scratch) | adjacent block's BS terms]
        auto row_dot = [&](const T *row, int r) -> T {
            T acc = pscr[r];
#pragma unroll
            for (int b = 0; b < BS; ++b) acc += row[2 * W + b] * xJ[b];
            return acc;
        };
        if constexpr (BS == 2) {
            const int r0 = tail ? 2 * N - gr.tu : 0;
            if (S == 32) {
                // one row per lane (m <= HMAX < 32); every operand is read before xJ arrives,
                // and alpha by every lane before any lane writes v' over it
                const int q = ls;
                const bool has = q < m;
                const int i = r0 + (has ? q : 0);
                const bool is_g = (i == 0) || (i == 2 * N - 1) || (i % 2 == 0);
                const int node = i == 0 ? 0 : (i == 2 * N - 1 ? N : (i + 1) / 2);
                const T *row = et + E::HZ + (has ? q : 0) * Z;
                const T base = pscr[has ? q : 0], k0 = row[2 * W], k1 = row[2 * W + 1];
                const T al = sA[node], vv = sV[node], pp = sP[node];
                const T x = base + k0 * xJ[0] + k1 * xJ[1];
                if (stage_v) __syncwarp();
                if (has) {
                    if (is_g) {
                        out_v(node, vv, beta, x);
                    } else {
                        const T ae = al * x;
                        out_p(node, pp - T(2) * ae, pp - ae);
                        if (node == src_k) add_source();
                    }
                }
                return;
            }
            // one row per lane (m <= 13 < S when v' is staged): alpha is read by every lane
            // before any lane writes v' over it
            for (int q0 = 0; q0 < m; q0 += S) {
                const int q = q0 + ls;
                const bool has = q < m;
                const int i = r0 + (has ? q : 0);
                const bool is_g = (i == 0) || (i == 2 * N - 1) || (i % 2 == 0);
                const int node = i == 0 ? 0 : (i == 2 * N - 1 ? N : (i + 1) / 2);
                const T x = has ? row_dot(et + E::HZ + q * Z, q) : T(0);
                const T al = sA[node];
                if (stage_v) __syncwarp();
                if (!has) continue;
                if (is_g) {
                    out_v(node, sV[node], beta, x);
                } else {
                    const T ae = al * x;
                    out_p(node, sP[node] - T(2) * ae, sP[node] - ae);
                    if (node == src_k) add_source();
                }
            }
        } else {
            const int cell0 = tail ? N - gr.tu + 1 : 1;
            const int qb = gr.mid + 3 * ((cg - c + tact) * MM - 1);  // first cell of the last middle block
            const int jlo = tail ? qb + 1 : 0, nrow = tail ? N - qb : gr.hu + 2;
            if (S == 32) {
                // one row per lane: pressure rows on lanes 0..15 (m <= HMAX), velocity rows on
                // lanes 16..31 (nrow <= HMAX + 2)
                static_assert(E::HMAX + 2 <= 16, "end rows fit a half-warp");
                const bool vel = ls >= 16;
                const int q = vel ? ls - 16 : ls;
                const bool has = q < (vel ? nrow : m);
                const int qq = has ? q : 0;
                const T x = row_dot(et + (vel ? E::DZ : E::HZ) + qq * Z, vel ? E::HMAX + qq : qq);
                if (has) {
                    if (vel) {
                        out_v(jlo + qq, sV[jlo + qq], beta * ih, x);
                    } else {
                        const int cc = cell0 + qq;
                        out_p(cc, T(2) * x - sP[cc], x);
                        if (cc == src_k) add_source();
                    }
                }
                return;
            }
            for (int q = ls; q < m; q += S) {
                const T x = row_dot(et + E::HZ + q * Z, q);
                const int cc = cell0 + q;
                out_p(cc, T(2) * x - sP[cc], x);
                if (cc == src_k) add_source();
            }
            for (int q = ls; q < nrow; q += S) {
                const int j = jlo + q;
                out_v(j, sV[j], beta * ih, row_dot(et + E::DZ + q * Z, E::HMAX + q));
            }
        }
    };
    __syncwarp();  // scratch rows written by other lanes (lines within one warp, no scan barrier)
    if (head_seg) seg_end(false);
    if (tail_seg) seg_end(true);
    // staged outputs are written to global memory by the staging warp once every compute warp
    // has released the stage; make this thread's shared-memory writes visible to those copies
    if (stage_v) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ---------------------------------------------------------------------------------------
// The kernel: persistent CTAs walk the line groups g = blockIdx.x, blockIdx.x + gridDim.x, ...
// through a ring of `stages` shared-memory stages.  The last warp stages the groups: one lane
// waits until the compute warps have released a stage (mbarrier "empty") and starts the bulk
// copies of the next group into it (mbarrier "full").  The 15 compute warps wait for "full",
// solve the group and release the stage.  Every wait is bounded; one that runs out sets *fault
// and the warp carries on with the same iteration count, so no warp is left waiting at a
// barrier and the launch ends (with garbage results and the fault flag set).
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ void mbar_arrive(unsigned long long *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

template <typename T, int BS, int MM, bool SPLIT, int NT>
__global__ void __launch_bounds__(NT, 1)
line_solve_factored_kernel(const LineDesc<T> *__restrict__ descs, const FacGroup *__restrict__ groups, int ngroups,
                           int natural, unsigned stage_bytes, int stages, int q, int *fault) {
    extern __shared__ __align__(128) unsigned char fac_smem[];
    __shared__ ScanSmem<T, BS> ssm;
    __shared__ __align__(8) unsigned long long full[kFacMaxStages], empty[kFacMaxStages];
    // chunk offsets of the windowed scans: forward and backward buffers for FP32, one for FP64
    constexpr int kBufs = sizeof(T) == 4 ? 2 : 1;
    __shared__ T offs[kBufs][NT * BS];
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) {
        for (int k = 0; k < kFacMaxStages; ++k) {
            mbar_init(&full[k], 1);
            mbar_init(&empty[k], (NT - 32) / 32);
        }
        mbar_fence_init();
    }
    __syncthreads();
    // the it-th group of this CTA goes to stage it % stages, as that stage's use-th group
    if (tid >= NT - 32) {  // the staging warp; every lane runs the same loop
        int last[kFacMaxStages];
        for (int k = 0; k < kFacMaxStages; ++k) last[k] = -1;
        int st = 0, use = 0;
        for (int gi = blockIdx.x; gi < ngroups; gi += gridDim.x) {
            unsigned char *stage = fac_smem + (size_t)st * stage_bytes;
            if (use > 0) {
                // the previous group of this stage is solved: write its outputs, then refill.
                // The copies that filled it have landed (the compute warps waited for them);
                // if a compute warp's wait ran out they may not have, so every lane waits for
                // them itself before it copies anything into the stage again.
                if (!mbar_wait(&empty[st], (unsigned)((use - 1) & 1))) atomicExch(fault, 1);
                if (!mbar_wait(&full[st], (unsigned)((use - 1) & 1))) atomicExch(fault, 1);
                fac_store_outputs<T>(stage, lane);
                __syncwarp();  // every lane's output copies have read the stage
            }
            fac_issue<T, BS, SPLIT>(descs, groups + gi, stage, &full[st], lane, q);
            last[st] = use;
            if (++st == stages) { st = 0; ++use; }
        }
        // the last groups of each stage: wait until solved and until their copies have
        // landed (no bulk copy into this CTA's shared memory may outlive it), write outputs
        for (int k = 0; k < stages; ++k)
            if (last[k] >= 0) {
                if (!mbar_wait(&empty[k], (unsigned)(last[k] & 1))) atomicExch(fault, 1);
                if (!mbar_wait(&full[k], (unsigned)(last[k] & 1))) atomicExch(fault, 1);
                fac_store_outputs<T>(fac_smem + (size_t)k * stage_bytes, lane);
            }
        // global visibility of this lane's output copies before the CTA ends
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        return;
    }
    int st = 0, use = 0;
    for (int gi = blockIdx.x; gi < ngroups; gi += gridDim.x) {
        if (!mbar_wait(&full[st], (unsigned)(use & 1))) atomicExch(fault, 1);
        fac_group<T, BS, MM, SPLIT, NT>(fac_smem + (size_t)st * stage_bytes, natural, ssm, offs[0], offs[kBufs - 1]);
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[st]);
        if (++st == stages) { st = 0; ++use; }
    }
}

// The records of nlines lines of one simulation and direction (N cells each).  dB: 18 FP64 values a line.
template <typename T>
cudaError_t launch_fac_precompute(const LineDesc<T> *d, int nlines, int method, int N, double *dB, int *status,
                                  cudaStream_t s) {
    if (nlines <= 0) return cudaSuccess;
    const int jobs = 2 * nlines;
    fac_ends_kernel<T><<<(jobs + kFacEndWarps - 1) / kFacEndWarps, 32 * kFacEndWarps, 0, s>>>(d, nlines, dB, status);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const FacGeom g = fac_geom(method, N);
    // threads per line: a power of two, up to four warps an SM in all (the FP64 pipe's four parts) while a run
    // is no shorter than half its warm-up (1023 CFD lines of 1024 cells: 267 us)
    int segs = 1, dev = 0, sms = 152;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        sms = 152;
    while (segs < 32 && (long long)nlines * segs < 4ll * 32 * sms && g.nb / (2 * segs) >= fac_warm(method) / 2) segs *= 2;
    const int per = kFacRecThreads / segs;
    fac_records_kernel<T><<<(nlines + per - 1) / per, kFacRecThreads, 0, s>>>(d, nlines, segs, dB, status);
    return cudaGetLastError();
}

template <typename T, int BS, int MM, bool SPLIT, int NT>
cudaError_t launch_fac_inst(const LineDesc<T> *d, const FacGroup *groups, int ngroups, size_t stage_bytes, int stages,
                            int grid, int natural, int q, int *fault, cudaStream_t s) {
    auto kern = line_solve_factored_kernel<T, BS, MM, SPLIT, NT>;
    // the host sizes the ring with fac_static_smem, an upper bound of the kernel's own static
    // shared memory: check it against the compiled kernel once.  The dynamic limit is the process's, so it is
    // all that the static part leaves, whatever this launch needs: no thread lowers it under another's launch
    static const int dyn_max = [&] {
        cudaFuncAttributes a{};
        if (cudaFuncGetAttributes(&a, kern) != cudaSuccess || a.sharedSizeBytes > fac_static_smem(sizeof(T), BS)) return -1;
        return (int)(kFacSmemLimit - a.sharedSizeBytes);
    }();
    const size_t dyn = (size_t)stages * stage_bytes;
    if (dyn_max < 0 || dyn > (size_t)dyn_max) return cudaErrorInvalidConfiguration;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn_max);
    if (e != cudaSuccess) return e;
    kern<<<grid, NT, dyn, s>>>(d, groups, ngroups, natural, (unsigned)stage_bytes, stages, q, fault);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_line_solve_factored(const LineDesc<T> *d, const FacGroup *groups, int ngroups, int variant,
                                       size_t stage_bytes, int stages, int grid, int natural, int q, int *fault,
                                       cudaStream_t s) {
    if (ngroups <= 0) return cudaSuccess;
    if (grid > ngroups) grid = ngroups;
    if (stages < 1 || stages > kFacMaxStages) return cudaErrorInvalidValue;
    constexpr int W = kFacThreads;
    switch (variant) {
    case 0: return launch_fac_inst<T, 2, 9, false, W>(d, groups, ngroups, stage_bytes, stages, grid, natural, q, fault, s);
    case 1: return launch_fac_inst<T, 3, 2, false, W>(d, groups, ngroups, stage_bytes, stages, grid, natural, q, fault, s);
    case 2: return launch_fac_inst<T, 3, 3, false, W>(d, groups, ngroups, stage_bytes, stages, grid, natural, q, fault, s);
    case 3: return launch_fac_inst<T, 2, 9, true, W>(d, groups, ngroups, stage_bytes, stages, grid, natural, q, fault, s);
    case 4: return launch_fac_inst<T, 3, 3, true, W>(d, groups, ngroups, stage_bytes, stages, grid, natural, q, fault, s);
    }
    if constexpr (sizeof(T) == 8) {
        constexpr int NR = kFacNarrow;
        switch (variant) {
        case 5: return launch_fac_inst<T, 3, 2, false, NR>(d, groups, ngroups, stage_bytes, stages, grid, natural, q, fault, s);
        case 6: return launch_fac_inst<T, 3, 3, false, NR>(d, groups, ngroups, stage_bytes, stages, grid, natural, q, fault, s);
        }
    }
    return cudaErrorInvalidValue;
}

template cudaError_t launch_fac_precompute<float>(const LineDesc<float> *, int, int, int, double *, int *, cudaStream_t);
template cudaError_t launch_fac_precompute<double>(const LineDesc<double> *, int, int, int, double *, int *, cudaStream_t);
template cudaError_t launch_line_solve_factored<float>(const LineDesc<float> *, const FacGroup *, int, int, size_t, int,
                                                       int, int, int, int *, cudaStream_t);
template cudaError_t launch_line_solve_factored<double>(const LineDesc<double> *, const FacGroup *, int, int, size_t,
                                                        int, int, int, int, int *, cudaStream_t);

// The bounded wait's failure path, run on purpose: one thread waits on an mbarrier that
// nothing arrives at, with `polls` polls at most, and records whether the wait gave up (and
// the time it took).  No other thread or copy is involved, so the kernel always ends.
__global__ void wait_timeout_probe_kernel(int polls, int *gave_up, long long *cycles) {
    __shared__ __align__(8) unsigned long long bar;
    if (threadIdx.x != 0) return;
    mbar_init(&bar, 1);
    mbar_fence_init();
    const long long t0 = clock64();
    const bool ok = mbar_wait(&bar, 0u, polls);
    *cycles = clock64() - t0;
    *gave_up = ok ? 0 : 1;
}

}  // namespace adi

extern "C" int adi_selftest_wait_timeout(int polls, int *gave_up, long long *cycles) {
    if (polls < 1 || polls > (1 << 22) || !gave_up) return ADI_EINVAL;
    int *d_flag = nullptr;
    long long *d_cyc = nullptr;
    cudaError_t e = cudaMalloc(&d_flag, sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&d_cyc, sizeof(long long));
    if (e == cudaSuccess) {
        adi::wait_timeout_probe_kernel<<<1, 32>>>(polls, d_flag, d_cyc);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(gave_up, d_flag, sizeof(int), cudaMemcpyDeviceToHost);
    long long c = 0;
    if (e == cudaSuccess) e = cudaMemcpy(&c, d_cyc, sizeof(long long), cudaMemcpyDeviceToHost);
    if (cycles) *cycles = c;
    if (d_flag) cudaFree(d_flag);
    if (d_cyc) cudaFree(d_cyc);
    if (e != cudaSuccess) { (void)cudaGetLastError(); return e == cudaErrorNoDevice ? ADI_ENOTSUP : ADI_ECUDA; }
    return ADI_OK;
}
