"""Host parts of the library, compiled by themselves and run without a GPU."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def run_native(tmp_path, source, *more, stdin=None):
    """Compiles tests/native/<source> (and the sources in `more`) against the CUDA headers, runs it, returns its output."""
    from paper_2609_02652_b200 import build

    cuda = os.path.join(os.path.dirname(os.path.dirname(build._tool("nvcc", "/usr/local/cuda/bin/nvcc"))), "include")
    exe = str(tmp_path / "a.out")
    subprocess.run([shutil.which("g++") or "/usr/bin/g++", "-O2", "-std=c++17", "-pthread", "-isystem", cuda, os.path.join(HERE, "native", source), *more, "-o", exe],
                   check=True, timeout=600)
    r = subprocess.run([exe], input=stdin, capture_output=True, text=stdin is None or isinstance(stdin, str), timeout=600)
    assert r.returncode == 0, (r.stdout[-2000:], r.stderr[-2000:])
    return r.stdout


def test_plan_cache_hands_out_whole_plans_to_threads(tmp_path):
    assert run_native(tmp_path, "plan_cache.cpp").strip() == "0"


def test_plan_of_five_to_eight_vectors(tmp_path):
    """The pass that llvq_gemv_plan does not describe (twelve warps, eight records of x a block): shares, panels, shared memory,
    and at most two panels' pieces of x a CTA on a full-size part, a thread each, so that none is read twice."""
    import numpy as np

    from paper_2609_02652_b200 import build

    build.build()
    rng = np.random.default_rng(12)
    shapes = [(148, 500, 8208, 5), (148, 2560, 9744, 5), (148, 1024, 17424, 8), (148, 1, 24, 6), (148, 36864, 5136, 7), (8, 4096, 98304, 8)]
    for _ in range(300):
        k = 24 * int(rng.integers(1, 4097) if rng.random() < 0.2 else rng.integers(1, 750))
        shapes.append((int(rng.choice([1, 8, 132, 148, 160, 320])), int(np.exp(rng.uniform(0, np.log(60000)))), k, int(rng.integers(5, 9))))
    where = os.path.dirname(build.LIB)
    out = run_native(tmp_path, "batch_plan.cpp", "-L" + where, "-l:libllvq.so", "-Wl,-rpath," + where, stdin="".join("%d %d %d %d\n" % s for s in shapes))
    lines = out.strip().splitlines()
    assert len(lines) == len(shapes)
    beyond = 0
    for (sm, rows, k, batch), line in zip(shapes, lines):
        grid, smem, units, panel, npanels, xblocks, groups, *ctas = map(int, line.split())
        nb, total, first = k // 24, groups * units, ctas[0::3]
        assert 1 <= grid <= min(sm, 256) and first[0] == 0 and first[-1] == total and all(a <= b for a, b in zip(first, first[1:]))
        assert 1 <= panel <= 16 and (npanels - 1) * panel < units <= npanels * panel
        for c in range(grid):
            f0, f1, lo, hi = first[c], first[c + 1], ctas[3 * c + 1], ctas[3 * c + 2]
            last = max(f1 - 1, f0)
            assert lo == min(f0 // (groups * panel), npanels - 1) * panel * 4
            assert hi == min(nb, (min(last // (groups * panel), npanels - 1) + 1) * panel * 4) and hi - lo <= xblocks
        assert smem >= 12 * 2 * 1792 + 8192 + 8 * xblocks * 112 + 12 * 2 * 8 + 12 * 4 * 8
        if sm >= 132:
            assert 3 * xblocks <= 12 * 32 and smem + 1024 <= 227 * 1024
        beyond += smem + 1024 > 227 * 1024
    assert beyond                     # few multiprocessors and a long row: the launch is refused, and llvq_gemv_batch takes two passes


def test_unranking_against_the_oracle(tmp_path, oracle):
    """Class, coordinates and window flags of indices at the edges of every class's digits: the tables and their readers, on the host."""
    import numpy as np

    from helpers import window_base
    from paper_2609_02652_b200 import build

    out = run_native(tmp_path, "unrank.cpp", *[os.path.join(build.CSRC, f) for f in ("llvq_tables.cpp", "llvq_unrank.cpp")], stdin=b"")
    r = np.frombuffer(out, np.dtype([("index", "<u8"), ("cls", "<u2"), ("window", "u1"), ("looked_at", "u1"), ("x", "i1", 24), ("pad", "u1", 4)]))
    assert np.unique(r["cls"]).size == 301 and r.size > 301 * 100
    x, cls = oracle.decode_batch(r["index"].copy())
    assert np.array_equal(r["cls"], cls) and np.array_equal(r["x"], x)
    none = window_base(x) == 0
    always, depends, never = 0, 1, 2
    assert not none[r["window"] == always].any() and none[r["window"] == never].all() and r["looked_at"][none].all()
    assert none[r["window"] == depends].any() and not none[r["window"] == depends].all()


def test_no_matvec_reads_ahead_of_an_expansion(tmp_path):
    """Every interleaving of two host threads' launches on one stream: the matvec on new records reads ahead in some of them, and never
    without an ordinary launch between it and the expansion."""
    total, ahead, wrong = map(int, run_native(tmp_path, "record_order.cpp").split())
    assert total == 462 and ahead > 0 and wrong == 0


def test_shares_cut_at_row_groups(tmp_path):
    """Every unit of a share is one warp's, a row group's sums are its own warps', and a CTA with a warp that ran into the wait limit hands nothing
    over: what lies in the place of that warp's sums is a record."""
    cuts, uncut, wrong = map(int, run_native(tmp_path, "cut.cpp").split())
    assert cuts > 10000 and uncut > 10000 and wrong == 0


def test_positions_of_pair_draws(tmp_path):
    """For every multiset, step and ratio the expander can meet, the position estimated for a pair's first and last rank is one of the pair's own or the
    next, never one before: the reader looks one entry back and no further."""
    from paper_2609_02652_b200 import build

    pairs, above, wrong = map(int, run_native(tmp_path, "pairs.cpp", *[os.path.join(build.CSRC, f) for f in ("llvq_tables.cpp", "llvq_unrank.cpp")]).split())
    assert pairs > 10000 and above > 0 and wrong == 0


def test_passes_of_a_batch(tmp_path):
    """A batch that one pass cannot carry goes in passes of four or of two, every vector in one of them and in order; what no pass can carry is
    refused with the size error, and another error ends it.  The plans of a device of few multiprocessors take every such way, those of a full-size one
    never more than one pass."""
    from paper_2609_02652_b200 import build

    build.build()
    where = os.path.dirname(build.LIB)
    shapes = [(sm, rows, 24 * nb, batch) for sm, rows in ((8, 4096), (8, 500), (1, 64), (148, 4096), (148, 33)) for nb in (70, 340, 355, 380, 500, 700, 4094) for batch in range(1, 9)]
    out = run_native(tmp_path, "passes.cpp", "-L" + where, "-l:libllvq.so", "-Wl,-rpath," + where, stdin="".join("%d %d %d %d\n" % s for s in shapes))
    counts, *lines = out.strip().splitlines()
    launched, refused, wrong = map(int, counts.split())
    assert launched > 100 and refused > 50 and wrong == 0 and len(lines) == len(shapes)
    seen = set()
    for (sm, _, _, batch), line in zip(shapes, lines):
        *passes, rc = map(int, line.split())
        assert rc == -3 or sum(passes) == batch
        assert sm < 148 or passes == [batch]
        seen.add(tuple(passes))
    assert {(4,), (2, 2), (2, 1), (8,), (4, 4), (2, 2, 2, 2)} <= seen
