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
