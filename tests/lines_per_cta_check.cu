// Host-only check of the stage's size: the lines that a CTA of the factored solver takes together at the lengths where they
// just fit its shared memory (one line fewer makes a launch of 704 lines two rounds of groups instead of one).  The
// counts follow from 227 KB a CTA less the static part's bound, two stages of a 128-byte group header, 208 bytes a line of
// descriptor (padded to 128) and the lines.  Built with nvcc and run on the host by tests/test_records.py; it launches no kernel.
#include "../paper_2006_07583_gb300/csrc/adi_factored.cu"
#include <cstdio>
using namespace adi;

int main() {
    int bad = 0;
    const struct { int method, n0, n1; size_t esz; int lines; } want[] = {
        {kCFD, 122, 122, 4, 24}, {kCFD, 39, 40, 8, 18}, {kCFD, 927, 930, 8, 3}, {kMFD, 147, 150, 4, 13}, {kMFD, 703, 706, 4, 5}};
    for (auto &w : want)
        for (int n = w.n0; n <= w.n1; ++n) {
            const int got = fac_lines_per_cta(w.method, n, w.esz);
            if (got != w.lines) { printf("FAIL method %d N %d: %d lines a CTA, not %d\n", w.method, n, got, w.lines); ++bad; }
        }
    printf("bad %d\n", bad);
    return bad != 0;
}
