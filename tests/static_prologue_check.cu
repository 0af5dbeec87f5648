// Host-only check of the windows that adi_step_static's prologue solves (prologue_win_rows with pivots), for every line of
// 16 to 128 cells: their error against an elimination in extended precision, over all lengths, is no larger than that of a
// plain elimination of the whole line in the same precision, each row's factors formed as it goes and divided by its
// pivot (but for 1 %: the two round the same rows differently).  Built with nvcc and run on the host by
// tests/test_prologue_rows.py; it launches no kernel.
#include "../paper_2006_07583_gb300/csrc/adi_kernels.cu"
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <vector>
using namespace adi;

// The tridiagonal rows and the right-hand sides in T of P g = Q u / h or Pbar e = Qbar w / h.
template <typename T>
struct System {
    int n;
    std::vector<double> lo, di, up;
    std::vector<T> q;
    System(int N, bool bar, const T *b, T ih) : n(bar ? N - 1 : N + 1), lo(n), di(n), up(n), q(n) {
        for (int r = 0; r < n; ++r) {
            double w[8], c[8];
            int c0 = 0, q0 = 0;
            const int len = bar ? cfd_Pbar_row(N, r + 1, &c0, w) : cfd_P_row(N, r, &c0, w);
            for (int i = 0; i < len; ++i) {
                const int col = (bar ? c0 - 1 : c0) + i;
                (col < r ? lo : (col > r ? up : di))[r] = w[i];
            }
            const int cnt = bar ? cfd_Qbar_row(N, r + 1, &q0, c) : cfd_Q_row(N, r, &q0, c);
            T acc = T(0);
            for (int t = 0; t < cnt; ++t) acc = std::fma((T)c[t], b[q0 + t], acc);
            q[r] = acc * ih;
        }
    }
    template <typename R>
    std::vector<R> eliminate() const {
        std::vector<R> cs(n), x(n);
        R c = 0, d = 0;
        for (int r = 0; r < n; ++r) {
            const R den = std::fma(-(R)lo[r], c, (R)di[r]);
            cs[r] = c = (R)up[r] / den;
            x[r] = d = std::fma(-(R)lo[r], d, (R)q[r]) / den;
        }
        for (int r = n - 2; r >= 0; --r) x[r] = std::fma(-cs[r], x[r + 1], x[r]);
        return x;
    }
};

template <typename T>
struct Rows {
    const std::vector<T> &q;
    void start(int) {}
    void next(int r, T (&v)[kProU]) { for (int i = 0; i < kProU; ++i) v[i] = r + i < (int)q.size() ? q[r + i] : T(0); }
    void back_start(int) {}
    void back(int, T (&)[kProU]) {}
};

template <typename T>
static int check(const char *name) {
    long double mine = 0, plain = 0;
    std::vector<double> f;
    unsigned seed = 12345;
    auto rnd = [&] { seed = seed * 1664525u + 1013904223u; return (double)(seed >> 8) / (1 << 24); };
    for (int N = 16; N <= 128; ++N)
        for (int bar = 0; bar < 2; ++bar)
            for (int rep = 0; rep < 40; ++rep) {
                std::vector<T> b(N + 1);
                double k[3], a[3];
                for (int m = 0; m < 3; ++m) { k[m] = 1 + (int)(rnd() * (N / 6)); a[m] = 2 * rnd() - 1; }
                for (int j = 0; j <= N; ++j) {
                    double v = 0;
                    for (int m = 0; m < 3; ++m) v += a[m] * (bar ? std::cos(M_PI * k[m] * j / N) : std::sin(M_PI * k[m] * j / N));
                    b[j] = (T)v;
                }
                const System<T> s(N, bar, b.data(), T(0.1));
                f.assign(prologue_factor_count(N), 0.0);
                prologue_factors(N, f.data(), true);
                const std::vector<T> ft(f.begin(), f.end());
                const T *fac = ft.data() + (bar ? 3 * (N + 1) : 0), *su = ft.data() + 3 * (N + 1) + 3 * (N - 1);
                std::vector<T> x(s.n);
                T tmp[kProR], halo[kProR];
                for (int r0 = 0; r0 < s.n; r0 += kProR) {
                    const int r1 = std::min(s.n, r0 + kProR);
                    if (prologue_inner(s.n, r0, r1)) { printf("FAIL N %d: a window without a boundary row\n", N); return 1; }
                    prologue_win_rows<false, T, true>(s.n, r0, r1, Rows<T>{s.q}, fac + r0, fac + s.n + r0, fac + 2 * s.n + r0,
                                                      su, tmp, halo, 1, [&](int r, T v, T) { x[r] = v; });
                }
                const std::vector<long double> ref = s.template eliminate<long double>();
                const std::vector<T> p = s.template eliminate<T>();
                long double nrm = 0, em = 0, ep = 0;
                for (int r = 0; r < s.n; ++r) {
                    nrm += ref[r] * ref[r];
                    em += (x[r] - ref[r]) * (x[r] - ref[r]);
                    ep += (p[r] - ref[r]) * (p[r] - ref[r]);
                }
                mine += em / nrm;
                plain += ep / nrm;
            }
    const double ratio = (double)std::sqrt(mine / plain);
    printf("%s: error over the plain elimination's %.4f\n", name, ratio);
    return !(ratio <= 1.01);
}

int main() {
    const int bad = check<float>("float") + check<double>("double");
    printf("bad %d\n", bad);
    return bad != 0;
}
