"""Shared memory of a pass of three or four vectors: on a full-size part it always fits; on a part of few multiprocessors, where a CTA's
records of x may not, it is beyond what passes in pairs of vectors needed by 32 bytes a block of x and no more, the margin
within which llvq_gemv_batch takes two passes."""
import os

import numpy as np

from test_native_cpu import run_native


def test_records_of_three_and_four_vectors(tmp_path):
    from paper_2609_02652_b200 import build

    build.build()
    rng = np.random.default_rng(31)
    shapes = [(148, 1, 24, 3), (148, 1024, 98256, 4), (8, 4096, 8160, 4), (1, 64, 24 * 340, 4)]
    for _ in range(300):
        shapes.append((int(rng.choice([1, 8, 16, 132, 148])), int(np.exp(rng.uniform(0, np.log(60000)))), 24 * int(rng.integers(1, 1500)), int(rng.integers(3, 5))))
    where = os.path.dirname(build.LIB)
    out = run_native(tmp_path, "batch_plan.cpp", "-L" + where, "-l:libllvq.so", "-Wl,-rpath," + where, stdin="".join("%d %d %d %d\n" % s for s in shapes))
    lines = out.strip().splitlines()
    assert len(lines) == len(shapes)
    margin = 0
    for (sm, rows, k, batch), line in zip(shapes, lines):
        smem, xblocks = int(line.split()[1]), int(line.split()[5])
        pairs = 16 * 2 * 1792 + 8192 + 8192 + (448 * xblocks + 127) // 128 * 128 + 16 * 2 * 8 + 16 * 4 * 4 + 16
        assert smem - 32 * xblocks <= pairs
        margin += smem + 1024 > 227 * 1024 >= pairs + 1024
        if sm >= 132:
            assert smem + 1024 <= 227 * 1024
    assert margin                        # some shape goes in two passes
