"""How the recomputed product is cut into blocks (fused_split, host): every
column is in a part, rows and columns stay within the kernel's limits, small
products get as many blocks as their rows and columns allow (up to 608, four
per SM), and products that fill the GPU with full tiles keep them.  Compiled
from the library's own plan source, as the plan check is."""
import os
import shutil
import subprocess

import pytest

from paper_2312_00005_gb300 import bemfmm

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_blocks_of_the_recomputed_product(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    bemfmm.lib()
    so = os.path.join(ROOT, "paper_2312_00005_gb300", "_bemfmm.so")
    exe = str(tmp_path / "fused_split_check")
    r = subprocess.run([cxx, "-O1", "-std=c++17", "-I/usr/local/cuda/include",
                        os.path.join(ROOT, "tests", "fused_split_check.cpp"),
                        os.path.join(ROOT, "paper_2312_00005_gb300", "csrc", "bem_plan.cpp"), so,
                        "-Wl,-rpath," + os.path.dirname(so), "-lpthread", "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    sizes = [1, 3, 4, 20, 31, 33, 80, 257, 320, 720, 1280, 2240, 2880, 5120, 9680, 40500, 2000000]
    pairs = [(n, c) for n in sizes for c in (1, n, 3200)]
    out = subprocess.run([exe] + [str(v) for p in pairs for v in p], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0
    for (n, c), line in zip(pairs, out.stdout.split("\n")):
        rows, cols, parts = map(int, line.split())
        assert rows in (4, 8, 16, 32) and cols in (32, 64, 128, 256) and parts >= 1, (n, c, line)
        tiles = -(-c // cols)
        assert parts <= max(1, tiles), (n, c, line)
        blocks = -(-n // rows) * parts
        if cols < 256:
            assert parts == tiles and -(-n // 32) * -(-c // 256) < 608
            assert blocks >= min(608, -(-n // 4) * -(-c // 32)) and blocks < 4 * 608, (n, c, line)
        else:
            assert rows == 32 and blocks <= max(3648, -(-n // 32)), (n, c, line)
