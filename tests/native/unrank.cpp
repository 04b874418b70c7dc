// The expander's un-ranking, run on the host: for indices at the edges of every class's digits and random ones between, a record
// of {index, class, window flag, whether the count looks at the index's slot, 24 coordinates} each on the standard output.
#include <cstdio>
#include <random>
#include <vector>

#include "../../paper_2609_02652_b200/csrc/llvq_tables.h"
#include "../../paper_2609_02652_b200/csrc/llvq_unrank.cuh"

using namespace llvq;

struct Record {
    uint64_t index;
    uint16_t cls;
    uint8_t window, looked_at;
    int8_t x[24];
    uint8_t pad[4];
};

int main() {
    HostTables t;
    UnrankTables u;
    if (!build_tables(t) || !build_unrank_tables(t, u)) return 1;
    const UnrankView v = {u.blob.data(), u.blob.data(), u.pairs.data(), u.tail8.data(), u.tab_b.data()};
    std::mt19937_64 rng(5);
    std::vector<uint64_t> indices;
    for (int c = 0; c < t.num_classes; c++) {
        const ClassDesc &d = t.desc[(size_t)c];
        const uint64_t first = t.base[(size_t)c], size = t.base[(size_t)c + 1] - first;
        auto add = [&](uint64_t at) { if (at < size) indices.push_back(first + at); };
        // the digits' steps: one, the signs or the message, the second arrangement, the first, the codeword
        const uint64_t digit = d.odd ? 4096 : 1ull << d.sign_bits, second = d.odd ? digit : digit * d.perm_b, top = d.odd ? digit : second * d.perm_a;
        add(0); add(size - 1);
        for (uint64_t step : {digit, second, top})
            for (int i = 0; i < 16; i++) {
                const uint64_t k = i < 4 ? (uint64_t)i + 1 : rng() % (size / step + 1);
                add(k * step); add(k * step - 1); add(k * step + 1);
            }
        for (int i = 0; i < 60; i++) add(rng() % size);
    }
    for (uint64_t index : indices) {
        Record r = {};
        r.index = index;
        const int c = find_class(v, index);
        const UnrankDesc d = blob_at<UnrankDesc>(v, kUnrankDescs, (uint32_t)c);
        const bool odd = d.flags & 1u;
        Point p;
        if (odd) unrank_odd(v, d, index - t.base[(size_t)c], p); else unrank_even(v, d, index - t.base[(size_t)c], p);
        r.cls = (uint16_t)c;
        r.window = (uint8_t)(d.flags >> 20);
        const int slot = guide_slot(index);
        r.looked_at = (uint8_t)(blob_at<uint32_t>(v, kUnrankWindow, (uint32_t)slot >> 5) >> (slot & 31) & 1u);
        for (int i = 0; i < 24; i++) r.x[i] = (int8_t)(2 * ((int)(point_codes(p, i >> 3, odd) >> (4 * (i & 7)) & 15u) - 8) + (odd ? 1 : 0));
        std::fwrite(&r, sizeof r, 1, stdout);
    }
    return 0;
}
