// The launch plan of a pass with more vectors than llvq_gemv_plan describes.  A line of input "sm rows k_padded batch" gives a
// line of output: grid, shared memory, units, panel, panels, blocks of x, row groups, then first unit and x blocks [lo, hi) of every CTA.
#include <cstdio>

#include "../../paper_2609_02652_b200/csrc/llvq_internal.cuh"

using namespace llvq;

int main() {
    int sm, rows, k, batch;
    while (std::scanf("%d %d %d %d", &sm, &rows, &k, &batch) == 4) {
        static GemvParams p;
        std::memset((void *)&p, 0, sizeof p);
        p.nprob = 1;
        p.batch = batch;
        p.nb = k / 24;
        p.tiles = p.nb / kTileCells;
        p.tail_cells = p.nb % kTileCells;
        p.units = p.tiles + (p.tail_cells ? 1 : 0);
        p.prob[0].rows = rows;
        p.total_groups = (rows + kRowsPerGroup - 1) / kRowsPerGroup;
        p.total_units = p.total_groups * p.units;
        const GemvLaunch g = gemv_plan(LLVQ_PLANES, p, sm);
        std::printf("%d %zu %d %d %d %d %d", g.grid, g.smem, p.units, p.panel, p.npanels, p.xblocks, p.total_groups);
        for (int c = 0; c < g.grid; c++) std::printf(" %d %d %d", p.cta[c].first, p.cta[c].blk_lo, p.cta[c].blk_hi);
        std::printf(" %d\n", p.cta[g.grid].first);
    }
    return 0;
}
