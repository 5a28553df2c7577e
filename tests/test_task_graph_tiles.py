"""The task graph with near tiles of 32 and 128 rows and doubled far tiles (the
heights a reordering chooses by its size and precision): the checks of
graph_check.cpp, compiled with a duration model that carries those heights."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1905_04975_gb300", "csrc")


@pytest.fixture(scope="module", params=[(32, 1), (128, 2)], ids=["near32", "near128"])
def checker(request, tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("graph")
    src = d / "check.cpp"
    src.write_text('#include "%s/host.h"\n'
                   "namespace gbr { struct Heights : CostModel { Heights() { near = %d; far_mul = %d; } }; }\n"
                   "#define CostModel Heights\n"
                   '#include "%s/tests/graph_check.cpp"\n' % (CSRC, *request.param, ROOT))
    subprocess.run([nvcc, "-O2", "-std=c++17", "-x", "cu", "-I", os.path.join(ROOT, "include"), str(src),
                    os.path.join(CSRC, "plan.cu"), "-o", str(d / "check")], check=True)
    return str(d / "check")


@pytest.mark.parametrize("n,w,m,q,z", [(40, 8, 3, 1, 0), (300, 64, 30, 1, 0), (257, 64, 32, 1, 1),
                                       (700, 128, 64, 1, 0), (900, 96, 40, 1, 0)])
def test_reordering_graph(checker, n, w, m, q, z):
    p = subprocess.run([checker] + [str(a) for a in (n, w, m, q, z, 3, 0)], capture_output=True, text=True,
                       timeout=300)
    assert p.returncode == 0 and p.stdout.startswith("OK"), p.stdout + p.stderr
