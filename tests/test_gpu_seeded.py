"""The FP64 building blocks that start from the special function unit's seeds
(seeded.cuh) and the sweep's reflector (sweep_body.cuh), at exact, tiny, huge
and random inputs, against values in extended precision.

Bounds, u = 2^-53.  rcp64: the seed's 2^-20 cubed is below 2^-59, and one
rounding follows: 1.1 u.  sqrt64: a residual correction of a value good to a few
u, one rounding: 1.1 u.  givens64: nn has two roundings that count half, 1 /
sqrt(nn) two more, the product one: 5 u.  Reflector: v1, v2 from a root, a sum, a
reciprocal and a product: 5 u; tau = 2 / (1 + v1^2 + v2^2) of the rounded v1,
v2, corrected: 1.5 u; beta as the root, after nn's roundings: 3 u.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1905_04975_gb300", "csrc")
LD = np.longdouble
U = 2.0 ** -53

SRC = """
#include "%s/sweep_body.cuh"
__global__ void k(int n, const double* a, double* o) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x = a[i], y = a[n + i], z = a[2 * n + i];
    o[i] = gbr::rcp64(x);
    o[n + i] = gbr::sqrt64(fabs(x));
    gbr::givens64(x, y, o + 2 * n + i, o + 3 * n + i);
    gbr::swp::refl3(3, x, y, z, o + 4 * n + i, o + 5 * n + i, o + 6 * n + i, o + 7 * n + i);
}
extern "C" int run(int n, const double* a, double* o) {
    k<<<(n + 127) / 128, 128>>>(n, a, o);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def values(tmp_path_factory):
    """x, y, z and the eight outputs, as columns."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not torch.cuda.is_available() or not os.path.exists(nvcc):
        pytest.skip("needs a GPU and nvcc")
    d = tmp_path_factory.mktemp("seeded")
    (d / "k.cu").write_text(SRC % CSRC)
    subprocess.run([nvcc, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-I", os.path.join(ROOT, "include"), "-shared",
                    "-Xcompiler", "-fPIC", "-o", str(d / "k.so"), str(d / "k.cu")], check=True)
    rng = np.random.default_rng(1)
    ex = [(0, 1, 0), (0, 0, 1), (0, .7, 0), (3, 4, 0), (-3, 0, 4), (1, 2, 2), (-2, 1, 2), (1, 0, 0), (2, 0, 0),
          (1, 1e-150, 1e-151), (1, 1e-154, 0), (1, 1e-155, 0), (4, 1e-155, 4e-155), (1e3, 1e-160, 1e-161),
          (1, 2.0 ** -26, 0), (1, 2.0 ** -27, 2.0 ** -27), (2.0 ** 400, 2.0 ** 399, 1), (2.0 ** -400, 2.0 ** -401, 0)]
    r = rng.standard_normal((20000, 3))
    r[5000:10000] *= 2.0 ** rng.integers(-60, 61, (5000, 3))
    r[10000:15000, 0] *= 2.0 ** rng.integers(-400, 401, 5000)
    r[10000:15000, 1:] = r[10000:15000, :1] * rng.standard_normal((5000, 2))
    r[15000:18000] = np.round(3 * r[15000:18000])
    r[18000:19000, 1] *= 1e-9  # almost no rotation
    r[19000:, 0] *= 1e-9       # almost an exchange
    x = np.concatenate([np.array(ex), r])
    x[:, 1] = np.where((x[:, 0] == 0) & (x[:, 1] == 0) & (x[:, 2] == 0), 1.0, x[:, 1])
    n = x.shape[0]
    a = torch.from_numpy(np.ascontiguousarray(x.T)).cuda()
    o = torch.zeros((8, n), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    lib = ctypes.CDLL(str(d / "k.so"))
    assert lib.run(n, ctypes.c_void_p(a.data_ptr()), ctypes.c_void_p(o.data_ptr())) == 0
    return x.T.astype(LD), o.cpu().numpy()


def rel(got, want):
    return np.max(np.abs(got.astype(LD) - want) / np.abs(want)) / LD(U)


def test_reciprocal_and_root(values):
    (x, _, _), o = values
    k = x != 0
    assert rel(o[0][k], 1 / x[k]) <= 1.1
    assert rel(o[1][k], np.sqrt(np.abs(x[k]))) <= 1.1


def test_rotation(values):
    (x, y, _), o = values
    k = (x != 0) | (y != 0)
    n = np.hypot(x[k], y[k])
    c, s = o[2][k].astype(LD), o[3][k].astype(LD)
    assert np.max(np.abs(c - x[k] / n)) <= 5 * U and np.max(np.abs(s - y[k] / n)) <= 5 * U


def test_rotation_by_almost_nothing(values):
    """Many such rotations are accumulated: their rounding errors must not have
    a mean.  The larger component is its correctly rounded value, 1; the other's
    square does not count."""
    (x, y, _), o = values
    for a, b in ((0, 1), (1, 0)):
        p = (x, y)
        k = np.abs(p[b]) * 2.0 ** 29 < np.abs(p[a])
        assert k.sum() > 500 and np.all(np.abs(o[2 + a][k]) == 1.0)


def test_reflector(values):
    (x, y, z), o = values
    v1, v2, tau, beta = (v.astype(LD) for v in o[4:])
    assert np.all(np.isfinite(o[4:]))
    sig = (o[4] != 0) | (o[5] != 0)          # a column that is not a multiple of e_0
    sq = y * y + z * z
    lost = sq.astype(np.float64) == 0.0      # its squares underflow: left as it is
    assert np.array_equal(sig | lost, (y != 0) | (z != 0) | lost)
    n = np.sqrt(x * x + sq)
    b = np.where(x >= 0, -n, n)
    d = x - b
    k = sig
    assert np.max(np.abs(v1[k] - y[k] / d[k])) <= 5 * U and np.max(np.abs(v2[k] - z[k] / d[k])) <= 5 * U
    assert rel(o[6][k], 2 / (1 + v1[k] ** 2 + v2[k] ** 2)) <= 1.5
    assert rel(o[7][k], b[k]) <= 3.0
    assert np.all(tau[~k] == 0) and np.array_equal(beta[~k], x[~k])
