"""Rows of the near update tiles by size, window and precision: half as high as
the default only where that was measured to be faster."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1905_04975_gb300", "csrc")
FMA, DMMA, SPLIT = "GBR_PREC_FMA", "GBR_PREC_DMMA", "GBR_PREC_OZAKI"
# n, window, precision, pair, rows
CASES = [(600, 128, FMA, 0, 32), (2500, 128, FMA, 0, 32), (4000, 128, FMA, 0, 64), (600, 72, FMA, 0, 32),
         (2500, 96, FMA, 0, 32),
         (2500, 72, FMA, 0, 64), (3000, 72, FMA, 0, 64), (1500, 64, FMA, 0, 64), (1500, 128, DMMA, 0, 32),
         (2500, 128, DMMA, 0, 64), (1500, 96, DMMA, 0, 64), (3000, 72, DMMA, 0, 64), (4000, 128, SPLIT, 0, 128),
         (2000, 64, FMA, 1, 32), (2400, 64, FMA, 1, 64), (800, 32, FMA, 1, 64), (2400, 16, FMA, 1, 64),
         (2000, 64, DMMA, 1, 64), (2400, 32, DMMA, 1, 64), (1000, 32, SPLIT, 1, 128)]


def test_near_tile_rows(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    calls = "".join("{ gbr::CostModel c; gbr::tile_heights(c, %d, %d, %s, %d); printf(\"%%d\\n\", c.near); }\n"
                    % (n, w, p, pair) for n, w, p, pair, _ in CASES)
    src = tmp_path / "heights.cpp"
    src.write_text('#include "%s/host.h"\n#include <stdio.h>\nint main() {\n%s}\n' % (CSRC, calls))
    subprocess.run([nvcc, "-std=c++17", "-x", "cu", "-I", os.path.join(ROOT, "include"), str(src), "-o",
                    str(tmp_path / "heights")], check=True)
    out = subprocess.run([str(tmp_path / "heights")], capture_output=True, text=True, check=True).stdout.split()
    got = [int(x) for x in out]
    assert got == [c[-1] for c in CASES], [c for c, g in zip(CASES, got) if c[-1] != g]
