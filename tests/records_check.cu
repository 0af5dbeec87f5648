// Host-only check of the factored records built by several runs a line (fac_run): a run that starts inside the line,
// fac_warm blocks early from G = 0, is kept only if it came to the G that the run before it ended with (fac_same_start).  The
// kept runs' records S, F and H are no further from the same records in extended precision, formed here from the blocks'
// definitions, than those of one run from the head (but for 10 %: the two round differently); constant, layered, random
// and smooth media, Courant numbers of 0.1 to 6.  At the usual Courant numbers every run is kept.  Built with nvcc and
// run on the host by tests/test_records.py; it launches no kernel.
#include "../paper_2006_07583_gb300/csrc/adi_factored.cu"
#include <cstdio>
#include <vector>
using namespace adi;
using LD = long double;

static unsigned long long g_seed;
static double uniform() {  // [0, 1)
    g_seed = g_seed * 6364136223846793005ULL + 1442695040888963407ULL;
    return (double)(g_seed >> 11) * 0x1p-53;
}

template <int BS>
struct Mat {
    LD m[BS][BS] = {};
    Mat operator*(const Mat &o) const {
        Mat r;
        for (int i = 0; i < BS; ++i)
            for (int j = 0; j < BS; ++j)
                for (int k = 0; k < BS; ++k) r.m[i][j] += m[i][k] * o.m[k][j];
        return r;
    }
    Mat neg() const {
        Mat r;
        for (int i = 0; i < BS; ++i)
            for (int j = 0; j < BS; ++j) r.m[i][j] = -m[i][j];
        return r;
    }
    Mat inverse() const {  // Gauss-Jordan, partial pivoting
        Mat a = *this, r;
        for (int i = 0; i < BS; ++i) r.m[i][i] = 1;
        for (int c = 0; c < BS; ++c) {
            int p = c;
            for (int i = c + 1; i < BS; ++i)
                if (fabsl(a.m[i][c]) > fabsl(a.m[p][c])) p = i;
            for (int j = 0; j < BS; ++j) { std::swap(a.m[c][j], a.m[p][j]); std::swap(r.m[c][j], r.m[p][j]); }
            const LD f = 1 / a.m[c][c];
            for (int j = 0; j < BS; ++j) { a.m[c][j] *= f; r.m[c][j] *= f; }
            for (int i = 0; i < BS; ++i) {
                if (i == c) continue;
                const LD x = a.m[i][c];
                for (int j = 0; j < BS; ++j) { a.m[i][j] -= x * a.m[c][j]; r.m[i][j] -= x * r.m[c][j]; }
            }
        }
        return r;
    }
};

// The records of a whole line in extended precision.
template <int BS>
static void exact(const LineDesc<double> &d, const FacGeom &g, const double *dB, std::vector<LD> &rec) {
    const size_t part = fac_part(g);
    const LD ih = d.inv_h, beta = d.beta;
    Mat<BS> G, F, H;
    for (int b = 0; b < g.nb; ++b) {
        Mat<BS> A, B, C;
        if (BS == 2) {
            const int j = g.first + b;
            const LD tb = 3 * beta * ih, am = 3 * ih * d.alpha[j - 1], ap = 3 * ih * d.alpha[j + 1];
            A.m[0][0] = A.m[1][1] = C.m[0][0] = C.m[1][1] = 1;
            B.m[0][0] = B.m[1][1] = 4;
            A.m[0][1] = -tb; A.m[1][0] = -am;
            C.m[0][1] = tb; C.m[1][0] = ap;
        } else {
            for (int m = 0; m < BS; ++m) {
                const LD sc = d.alpha[g.first + 3 * b + m] * beta * ih * ih;
                for (int q = 0; q < BS; ++q) {
                    A.m[m][q] = q >= m ? -sc * mim_DG(q - m) : 0;
                    B.m[m][q] = (q == m) - sc * mim_DG(q - m + 3);
                    C.m[m][q] = q <= m ? -sc * mim_DG(q - m + 6) : 0;
                }
            }
        }
        const bool first = b == 0, last = b == g.nb - 1;
        if (first) A = Mat<BS>();
        if (last) C = Mat<BS>();
        Mat<BS> S = A * G;
        for (int p = 0; p < BS; ++p)
            for (int q = 0; q < BS; ++q)
                S.m[p][q] = B.m[p][q] - S.m[p][q] - (first ? dB[p * BS + q] : 0) - (last ? dB[9 + p * BS + q] : 0);
        const Mat<BS> R = S.inverse(), E = (R * A).neg();
        G = R * C;
        const int c = b / g.mm, i = b % g.mm;
        F = i == 0 ? E : E * F;
        H = i == 0 ? G.neg() : (H * G).neg();
        for (int p = 0; p < BS; ++p)
            for (int q = 0; q < BS; ++q) {
                const size_t at = (size_t)c * BS * BS + p * BS + q;
                if (i == 0) rec[at] = S.m[p][q];
                rec[part + at] = F.m[p][q];
                rec[2 * part + at] = H.m[p][q];
            }
    }
}

template <int BS>
static int check(int method, const char *name) {
    int bad = 0;
    for (int kind = 0; kind < 4; ++kind)
        for (double cfl : {0.1, 0.2, 0.4, 0.8, 1.5, 3.0, 6.0}) {
            g_seed = 11;
            int kept = 0, runs = 0;
            LD es[3] = {}, eh[3] = {};
            for (int trial = 0; trial < 24; ++trial) {
                const int N = 700 + 97 * trial, warm = fac_warm(method);
                const FacGeom g = fac_geom(method, N);
                const double h = 1.0 / N, cmax = 1.4, dt = cfl * h / cmax, c0 = cmax * (0.3 + 0.7 * uniform());
                double layers[6];
                for (double &l : layers) l = cmax * (0.3 + 0.7 * uniform());
                std::vector<double> alpha(N + 2), rec(fac_rec(g)), head(fac_rec(g));
                for (int k = 0; k < N + 2; ++k) {
                    const double y = (double)k / (N + 1), r = uniform();
                    const double c = kind == 0 ? c0 : kind == 1 ? layers[(int)(5.999 * y)] : kind == 2 ? cmax * (1 - 0.4 * r)
                                                                                          : c0 * (1 + 0.1 * exp(-(y - 0.4) * (y - 0.4) / 0.02));
                    alpha[k] = 0.5 * dt * c * c;
                }
                LineDesc<double> d{};
                d.alpha = alpha.data();
                d.sp = 1;
                d.N = N;
                d.method = method;
                d.beta = 0.5 * dt;
                d.inv_h = 1.0 / h;
                double dB[18];
                for (double &x : dB) x = 0.2 * (uniform() - 0.5);
                double G[BS][BS] = {};
                if (!fac_run<double, true>(d, g, dB, dB + 9, head.data(), 0, g.nb, G)) { ++bad; continue; }
                std::vector<LD> ref(fac_rec(g));
                exact<BS>(d, g, dB, ref);
                int segs = 1;
                while (segs < 32 && g.nb / (2 * segs) >= warm / 2) segs *= 2;
                for (int seg = 1; seg < segs; ++seg) {
                    const int t0 = g.tact * seg / segs, t1 = g.tact * (seg + 1) / segs, b0 = t0 * g.mm;
                    double S[BS][BS] = {}, E[BS][BS] = {};
                    ++runs;
                    if (!fac_run<double, false>(d, g, dB, dB + 9, rec.data(), b0 > warm ? b0 - warm : 0, b0, S)) continue;
                    fac_run<double, false>(d, g, dB, dB + 9, rec.data(), 0, b0, E);
                    if (!fac_same_start(&S[0][0], &E[0][0], BS * BS)) continue;
                    ++kept;
                    fac_run<double, true>(d, g, dB, dB + 9, rec.data(), b0, t1 * g.mm, S);
                    for (int part = 0; part < 3; ++part) {
                        LD nr = 0, a = 0, b = 0;
                        for (int k = t0 * BS * BS; k < t1 * BS * BS; ++k) {
                            const size_t at = (size_t)part * fac_part(g) + k;
                            nr += ref[at] * ref[at];
                            a += (rec[at] - ref[at]) * (rec[at] - ref[at]);
                            b += (head[at] - ref[at]) * (head[at] - ref[at]);
                        }
                        if (nr > 0) { es[part] += a / nr; eh[part] += b / nr; }
                    }
                }
            }
            for (int part = 0; part < 3; ++part)
                if (!(es[part] <= 1.1 * 1.1 * eh[part])) {
                    printf("FAIL %s medium %d Courant %g record %d: error %.3Lf times that of one run\n", name, kind, cfl, part, sqrtl(es[part] / eh[part]));
                    ++bad;
                }
            if (cfl <= 1.0 && kept != runs) { printf("FAIL %s medium %d Courant %g: %d of %d runs kept\n", name, kind, cfl, kept, runs); ++bad; }
        }
    return bad;
}

int main() {
    const int bad = check<2>(kCFD, "CFD") + check<3>(kMFD, "MFD");
    printf("bad %d\n", bad);
    return bad != 0;
}
