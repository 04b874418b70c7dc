// Two host threads on one stream, every interleaving of their steps: one expands and then launches a matvec on the new records, the other
// launches two matvecs on records of its own.  How often may the first read its records ahead, and how often with no ordinary launch
// between it and the expansion (which must be never)?
#include <algorithm>
#include <cstdio>
#include <iterator>
#include <vector>

#include "../../paper_2609_02652_b200/csrc/llvq_internal.cuh"

using namespace llvq;

int main() {
    // an expansion's steps: enqueue, count; a matvec's: look, enqueue, settle
    int order[] = {0, 0, 0, 0, 0, 1, 1, 1, 1, 1, 1};
    long total = 0, ahead = 0, wrong = 0;
    do {
        RecordOrder r;
        std::vector<char> stream;              // x the expansion, o an ordinary launch, p a launch that reads ahead, P that of the new records
        uint64_t seen[2] = {0, 0};
        bool behind[2] = {false, false};
        int at[2] = {0, 0};
        for (int t : order) {
            const int step = at[t]++;
            if (t == 0 && step == 0) { stream.push_back('x'); continue; }
            if (t == 0 && step == 1) { r.expanded(); continue; }
            const int s = t == 0 ? step - 2 : step % 3;
            if (s == 0) { seen[t] = r.expansions(); behind[t] = r.behind(seen[t]); }
            else if (s == 1) stream.push_back(!behind[t] ? 'o' : (t == 0 ? 'P' : 'p'));
            else if (!behind[t]) r.ordered(seen[t]);
        }
        total++;
        const auto reader = std::find(stream.begin(), stream.end(), 'P');
        if (reader != stream.end()) {
            ahead++;
            wrong += std::find(std::find(stream.begin(), stream.end(), 'x'), reader, 'o') == reader;
        }
    } while (std::next_permutation(std::begin(order), std::end(order)));
    std::printf("%ld %ld %ld\n", total, ahead, wrong);
    return 0;
}
