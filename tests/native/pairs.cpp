// The expander's tables of pair draws, whole: for every multiset, every step and every ratio that leads there, the position estimated for the first and
// the last rank of each pair.  Between those the estimate ascends, so the two hold it for all ranks.  Then a table that names no rank, on which the
// reader has to end all the same, one entry back.  Prints the pairs looked at, the estimates that were one position too
// large, and those that were neither that nor right.
#include <cstdio>
#include <set>
#include <vector>

#include "../../paper_2609_02652_b200/csrc/llvq_tables.h"
#include "../../paper_2609_02652_b200/csrc/llvq_unrank.cuh"

using namespace llvq;

int main() {
    HostTables t;
    UnrankTables u;
    if (!build_tables(t) || !build_unrank_tables(t, u)) return 1;
    const UnrankView v = {u.blob.data(), u.blob.data(), u.pairs.data(), u.tail8.data(), u.tab_b.data()};
    std::vector<std::set<uint32_t>> ratios(kOddSets);                     // of this step, as a float's bits
    for (int c = 0; c < t.num_classes; c++) {
        const uint32_t flags = blob_at<uint32_t>(v, kUnrankFlags, (uint32_t)c), set = (flags >> 1) & 255u;
        if (flags & 1u) ratios[set].insert(float_bits(blob_at<float>(v, kUnrankRatio, set)));
    }
    long pairs = 0, above = 0, wrong = 0;
    size_t first = 0;
    for (int step = 0; step < kPairSteps; step++) {
        const uint32_t left = 24 - 2 * step, draws = left * (left - 1);
        std::vector<std::set<uint32_t>> next(kOddSets);
        for (int set = 0; set < kOddSets; set++) {
            if (ratios[set].empty()) continue;
            const uint64_t *entry = u.pairs.data() + first + (size_t)set * draws;
            // positions where a pair begins; ranks are in proportion to positions, which gives the number of orderings
            std::vector<uint32_t> begin;
            for (uint32_t at = 0; at < draws; at++)
                if (at == 0 || entry[at] != entry[at - 1]) begin.push_back(at);
            const uint32_t last = begin.back();
            const uint64_t orderings = last ? (uint64_t)(uint32_t)entry[last] * draws / last : 1;
            wrong += (uint32_t)entry[0] != 0;
            for (size_t i = 0; i < begin.size(); i++) {
                const uint32_t end = i + 1 < begin.size() ? begin[i + 1] : draws;
                const uint32_t r0 = (uint32_t)entry[begin[i]], r1 = (end < draws ? (uint32_t)entry[end] : (uint32_t)orderings) - 1u;
                for (uint32_t bits : ratios[set]) {
                    pairs++;
                    for (uint32_t r : {r0, r1}) {
                        const uint32_t at = draw_position(r, bits_float(bits), draws);
                        above += at == end;
                        wrong += at < begin[i] || at > end || pair_drawn(entry + at, r) != entry[begin[i]];
                    }
                }
                const uint32_t high = (uint32_t)(entry[begin[i]] >> 32);
                if (step + 1 < kPairSteps) next[high & 255u].insert((high >> 4) + kRatioBase);
            }
        }
        first += (size_t)kOddSets * draws;
        ratios.swap(next);
    }
    const uint64_t nowhere[3] = {7u, 0xffffffffu, 0xffffffffu};
    wrong += pair_drawn(nowhere + 2, 5u) != nowhere[1];
    std::printf("%ld %ld %ld\n", pairs, above, wrong);
    return first == u.pairs.size() ? 0 : 1;
}
