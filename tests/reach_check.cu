// Host-only check of the windowed scans' reach (fac_reach), which forms its products in FP32 and again in FP64 where FP32
// cannot decide: it equals the reach of the same products in FP64 throughout, for transfers that decay as ordinary lines' do,
// for ones whose products nearly cancel, and for norms around the threshold.  Built with nvcc and run on the host by
// tests/test_records.py; it launches no kernel.
#include "../paper_2006_07583_gb300/csrc/adi_factored.cu"
#include <cstdio>
#include <vector>
using namespace adi;

static unsigned long long g_seed = 7;
static double uniform() {  // [-1, 1)
    g_seed = g_seed * 6364136223846793005ULL + 1442695040888963407ULL;
    return (double)(g_seed >> 11) * 0x1p-52 - 1.0;
}

template <typename TS, int BS>
static int exact(const TS *maps, int tact, double tau, bool forward) {
    int reach = 0;
    bool unsure;
    for (int e = 0; e < tact - 1 && reach <= kFacMaxReach; ++e) {
        const int r = fac_window<TS, BS, double>(maps, tact, tau, forward, forward ? e : e + 1, unsure);
        reach = r > reach ? r : reach;
    }
    return reach;
}

template <typename TS, int BS>
static int check(const char *name) {
    const double tau = sizeof(TS) == 4 ? 0x1p-40 : 0x1p-70;
    const int tact = 40;
    int bad = 0;
    for (int kind = 0; kind < 4; ++kind)
        for (int trial = 0; trial < 2000; ++trial) {
            std::vector<TS> maps((size_t)tact * BS * BS);
            const double scale = kind == 3 ? 0.6 : exp2(-2.0 - 6.0 * (1 + uniform()));  // 3: beyond the windows
            for (int k = 0; k < tact; ++k)
                for (int p = 0; p < BS; ++p)
                    for (int q = 0; q < BS; ++q) {
                        TS &m = maps[(size_t)k * BS * BS + p * BS + q];
                        if (kind == 1) m = (TS)((p == 0 ? 1.0 : -1.0) * (p < 2 && q < 2) + 1e-9 * uniform());  // squares to nearly zero
                        else if (kind == 2) m = (TS)(p == q ? exp2(log2(tau) / (3 + trial % 4)) * (1 + 1e-5 * uniform()) : 0.0);  // near tau
                        else m = (TS)(scale * uniform());
                    }
            for (int forward = 0; forward < 2; ++forward) {
                const int want = exact<TS, BS>(maps.data(), tact, tau, forward);
                const int got = fac_reach<TS, BS>(maps.data(), tact, tau, forward, 0, tact);
                if (want != got && ++bad <= 4) printf("FAIL %s kind %d: reach %d, in FP64 %d\n", name, kind, got, want);
            }
        }
    return bad;
}

int main() {
    const int bad = check<float, 2>("float 2x2") + check<float, 3>("float 3x3") + check<double, 2>("double 2x2") + check<double, 3>("double 3x3");
    printf("bad %d\n", bad);
    return bad != 0;
}
