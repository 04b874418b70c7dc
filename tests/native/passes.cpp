// The passes that a batch of activation vectors takes where one for all of them is refused, with a pass that launches nothing: every number of vectors,
// every largest pass that fits and every pass that fails for another reason.  Prints the batches that were launched
// whole, those that were refused or failed, and the mistakes.  Then, for every line of input "sm rows k_padded batch", the passes that the plans for such a
// device give (the vectors of each, in order), or the error.
#include <cstdio>
#include <vector>

#include "../../paper_2609_02652_b200/csrc/llvq_internal.cuh"

using namespace llvq;

int main() {
    long launched = 0, refused = 0, wrong = 0;
    for (int batch = 1; batch <= LLVQ_MAX_BATCH; batch++)
        for (int fits = 0; fits <= LLVQ_MAX_BATCH; fits++)          // vectors of the largest pass that fits
            for (int fails_at = -1; fails_at < 4; fails_at++) {     // which launch meets another error, none: -1
                std::vector<int> carried(LLVQ_MAX_BATCH, 0);
                int passes = 0, next = 0;
                bool in_order = true;
                const int rc = batch_passes(batch, [&](int first, int n) -> int {
                    if (first < 0 || n < 1 || first + n > batch) { in_order = false; return LLVQ_EINVAL; }
                    if (n > fits) return n > 2 && n <= kVectorsPerPass && fits >= 2 ? kTwoByTwo : LLVQ_ESIZE;
                    if (passes++ == fails_at) return LLVQ_ECUDA;
                    in_order = in_order && first == next;
                    next = first + n;
                    for (int j = first; j < first + n; j++) carried[(size_t)j]++;
                    return LLVQ_OK;
                });
                const bool all = next == batch;
                for (int j = 0; j < batch && all; j++) wrong += carried[(size_t)j] != 1;
                wrong += !in_order;
                // one pass where it fits; else none larger than four; two vectors and one have no smaller pass
                const bool possible = fits >= batch || (batch > 2 && fits >= 2);
                if (rc == LLVQ_OK) { launched++; wrong += !all || !possible || (fits >= batch && passes != 1); }
                else { refused++; wrong += possible ? (rc != LLVQ_ECUDA || fails_at < 0) : rc != LLVQ_ESIZE; }
            }
    std::printf("%ld %ld %ld\n", launched, refused, wrong);

    int sm, rows, k, batch;
    while (std::scanf("%d %d %d %d", &sm, &rows, &k, &batch) == 4) {
        const int rc = batch_passes(batch, [&](int, int n) -> int {
            static GemvParams p;
            std::memset((void *)&p, 0, sizeof p);
            p.nprob = 1;
            p.batch = n;
            p.nb = k / 24;
            p.tiles = p.nb / kTileCells;
            p.tail_cells = p.nb % kTileCells;
            p.units = p.tiles + (p.tail_cells ? 1 : 0);
            p.prob[0].rows = rows;
            p.total_groups = (rows + kRowsPerGroup - 1) / kRowsPerGroup;
            p.total_units = p.total_groups * p.units;
            const GemvLaunch g = gemv_plan(LLVQ_PLANES, p, sm);
            const int refusal = pass_refusal(n, g.smem, p.xblocks, 227 * 1024);
            if (refusal == LLVQ_OK) std::printf("%d ", n);
            return refusal;
        });
        std::printf("%d\n", rc);
    }
    return 0;
}
