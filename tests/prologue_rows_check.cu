// Host-only check of the prologue kernel's row accessor (ProRows) and of its windows (prologue_win_rows, with
// and without the constant interior factors): over every line length from 16 to 4096 cells, each row that a window
// asks for lies inside the line's natural fields; and for some lengths, those around the first constant-factor
// window and a long one among them, every row is written once and the solutions of P x = Q u / h and
// Pbar x = Qbar w / h agree to 1e-13 with an elimination of the same App. A matrices in extended precision,
// assembled from their row functions.  Built with nvcc and run on the host by tests/test_prologue_rows.py; it launches
// no kernel.
#include "../paper_2006_07583_gb300/csrc/adi_kernels.cu"
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <vector>
using namespace adi;

static long long g_outside, g_first;  // reads outside the field; the first one's row beyond the last
// A field's values along one line, from row `off` on.
struct Field {
    const double *p;
    int size, off;
    double operator[](long long i) const {
        const long long k = off + i;
        if (k >= 0 && k < size) return p[k];
        if (!g_outside++) g_first = k < 0 ? k : k - size + 1;
        return 0.0;
    }
};

// One operator of a line of N cells (bar: Pbar), chunk by chunk as the kernel takes it.
static int solve(int N, bool bar, const double *u, const double *w, const double *fac, std::vector<double> &xs,
                 std::vector<double> &ys, std::vector<int> &hits) {
    const int n = bar ? N - 1 : N + 1;
    const double ih = 3.0;
    const double *f = fac + (bar ? 3 * (N + 1) : 0), *su = fac + 3 * (N + 1) + 3 * (N - 1), *b = bar ? w : u;
    const Field x{b, N + 1, bar ? 1 : 0}, y{bar ? u : w, N + 1, bar ? 1 : 0};
    auto boundary = [&](int j) {
        double c[8], acc = 0.0;
        int c0;
        const int cnt = bar ? cfd_Qbar_row(N, j, &c0, c) : cfd_Q_row(N, j, &c0, c);
        for (int t = 0; t < cnt; ++t) acc += c[t] * b[c0 + t];
        return acc * ih;
    };
    int inner = 0;
    double tmp[kProR], halo[kProR];
    auto out = [&](int r, double v, double yr) { xs[r] = v; ys[r] = yr; ++hits[r]; };
    for (int r0 = 0; r0 < n; r0 += kProR) {
        const int r1 = std::min(n, r0 + kProR), k0 = bar ? -1 : 0, k1 = bar ? N - 1 : N;
        if (prologue_inner(n, r0, r1)) {
            ProRows<double, true, Field> rows{x, y, 1, 1, 0, k1, n, r0, r1, ih};
            prologue_win_rows<true, double>(n, r0, r1, rows, f + r0, f + n + r0, f + 2 * n + r0, su, tmp, halo, 1, out);
            ++inner;
        } else {
            ProRows<double, false, Field> rows{x, y, 1, 1, k0, k1, n, r0, r1, ih};
            rows.first = r0 == 0 ? boundary(bar ? 1 : 0) : 0.0;
            rows.last = r1 + kProH >= n ? boundary(bar ? N - 1 : N) : 0.0;
            prologue_win_rows<false, double>(n, r0, r1, rows, f + r0, f + n + r0, f + 2 * n + r0, su, tmp, halo, 1, out);
        }
    }
    return inner;
}

// The same system by an elimination of the whole line in extended precision.
static std::vector<long double> whole(int N, bool bar, const double *b) {
    const int n = bar ? N - 1 : N + 1;
    std::vector<long double> up(n), d(n);
    long double c = 0, v = 0;
    for (int r = 0; r < n; ++r) {
        double w[8], q[8], lo = 0, di = 0, su = 0;
        int c0 = 0, q0 = 0;
        const int len = bar ? cfd_Pbar_row(N, r + 1, &c0, w) : cfd_P_row(N, r, &c0, w);
        for (int i = 0; i < len; ++i) {
            const int col = (bar ? c0 - 1 : c0) + i;
            (col < r ? lo : (col > r ? su : di)) = w[i];
        }
        const int cnt = bar ? cfd_Qbar_row(N, r + 1, &q0, q) : cfd_Q_row(N, r, &q0, q);
        long double rhs = 0;
        for (int t = 0; t < cnt; ++t) rhs += (long double)q[t] * b[q0 + t];
        const long double den = (long double)di - (long double)lo * c;
        c = up[r] = su / den;
        v = d[r] = (rhs * 3.0L - lo * v) / den;
    }
    for (int r = n - 2; r >= 0; --r) d[r] -= up[r] * d[r + 1];
    return d;
}

int main() {
    int bad = 0;
    std::vector<double> u(4097), w(4097), x(4097), y(4097), f;
    std::vector<int> hits(4097);
    for (int k = 0; k < 4097; ++k) {
        u[k] = std::sin(0.37 * k) + 0.5;
        w[k] = std::cos(0.71 * k) - 0.3 * std::sin(0.05 * k);
    }
    int lengths_outside = 0;
    for (int N = 16; N <= 4096; ++N) {
        prologue_factors(N, f);
        for (int bar = 0; bar < 2; ++bar) {
            const int n = bar ? N - 1 : N + 1;
            g_outside = 0;
            std::fill(hits.begin(), hits.end(), 0);
            const int inner = solve(N, bar, u.data(), w.data(), f.data(), x, y, hits);
            if (g_outside) {
                if (++lengths_outside <= 5) printf("FAIL N %d bar %d reads %lld values outside, the first %lld rows beyond\n", N, bar, g_outside, g_first);
                ++bad;
            }
            for (int r = 0; r < n; ++r)
                if (hits[r] != 1 || y[r] != (bar ? u[r + 1] : w[r])) { printf("FAIL N %d bar %d row %d\n", N, bar, r); ++bad; break; }
            if (N > 300 && N % 97 != 0 && N != 1001) continue;
            const std::vector<long double> xd = whole(N, bar, bar ? w.data() : u.data());
            long double err = 0, nrm = 0;
            for (int r = 0; r < n; ++r) { err = std::max(err, std::fabs(x[r] - xd[r])); nrm = std::max(nrm, std::fabs(xd[r])); }
            if (!(err <= 1e-13L * nrm)) { printf("FAIL N %d bar %d inner %d err %Lg of %Lg\n", N, bar, inner, err, nrm); ++bad; }
            if ((inner > 0) != (n > 2 * kProR + kProH)) { printf("FAIL N %d bar %d inner windows %d\n", N, bar, inner); ++bad; }
        }
    }
    printf("bad %d\n", bad);
    return bad != 0;
}
