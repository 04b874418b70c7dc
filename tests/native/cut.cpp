// Every division of a share of units over the warps of a CTA, as the batch kernel cuts it and adds the warps' sums up: the ranges
// cover the share and cross no row group, a row group's sums are those of its own warps, and of a CTA with a warp that gave up nothing is
// handed over.  Prints the shares that were cut, those that were not, and the mistakes.
#include <cstdio>
#include <random>
#include <vector>

#include "../../paper_2609_02652_b200/csrc/llvq_cut.h"

using namespace llvq;

int main() {
    std::mt19937 rng(3);
    long cuts = 0, uncut = 0, wrong = 0;
    for (int warps : {12, 16})
        for (int width = 1; width <= 24; width++)
            for (int before = 0; before < width; before++)         // units of the share's first row group that are not its own
                for (int n = 1; n <= 400; n++)
                    for (int most = (n + warps - 1) / warps; most <= (n + warps - 1) / warps + 1; most++) {
                        const int head = width - before < n ? width - before : n, rows = (n - head) / width;
                        Cut c;
                        if (!cut_share(5, head, rows, n - head - rows * width, width, most, warps, c)) { uncut++; continue; }
                        cuts++;
                        // a unit's sum is its number plus one; a warp that gave up has left something else
                        const int gave_up = rng() % 4 == 0 ? (int)(rng() % (unsigned)warps) : -1;
                        std::vector<long> sum((size_t)warps, 1000000007l);
                        int next = 0;
                        bool lost = false;
                        for (int w = 0; w < warps; w++) {
                            int at;
                            const int k = cut_range(c, n, most, w, at);
                            if (k == 0) continue;
                            wrong += at != next || k > most || (before + at) / width != (before + at + k - 1) / width;
                            next = at + k;
                            lost = lost || w == gave_up;
                            if (w == gave_up) continue;
                            sum[(size_t)w] = 0;
                            for (int u = at; u < at + k; u++) sum[(size_t)w] += u + 1;
                        }
                        wrong += next != n || c.first_group != 5 || c.groups != (before + n - 1) / width + 1;
                        for (int batch : {3, 4, 8}) {
                            const int outputs = cut_outputs(c, batch, lost);
                            wrong += outputs != (lost ? 0 : 32 * batch * c.groups);
                            for (int o = 0; o < outputs; o += 32) {
                                const int s = cut_ratio(o >> 5, batch), begin = s == 0 ? 0 : s * width - before;
                                const int end = (s + 1) * width - before < n ? (s + 1) * width - before : n;
                                long want = 0, got = 0;
                                for (int u = begin; u < end; u++) want += u + 1;
                                const CutWarps of = cut_warps(c, s);
                                for (int w = of.first; w < of.end; w++) got += sum[(size_t)w];
                                wrong += s != (o >> 5) / batch || got != want || cut_units(c, s) != end - begin;
                            }
                        }
                    }
    std::printf("%ld %ld %ld\n", cuts, uncut, wrong);
    return 0;
}
