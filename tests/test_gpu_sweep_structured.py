"""Sweeps on structured matrices, whose reflectors have columns with zeros and
small integers: 1 + v1^2 + v2^2 is then exact and its rounding error exactly
zero, or so small that squares leave the normal range.  What is asserted holds
for any backward stable sweep: finite, Hessenberg, Q orthogonal and
A = Q H Q^T within 50 n eps (the bound of the other sweep tests).  Where the
reflectors are exact (permutations), also the oracle's entries.
"""
import numpy as np
import pytest

import oracle
from tests.helpers import EPS, orth_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gbr():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1905_04975_gb300 as g
    g.load()
    return g


def hessenberg(kind, n):
    """H, shifts and whether all reflectors are permutations."""
    H = np.zeros((n, n), order="F")
    i = np.arange(n - 1)
    if kind == "second difference":      # the first reflector is of (0, 0, 1)
        H[np.arange(n), np.arange(n)] = 2.0
        H[i, i + 1] = H[i + 1, i] = -1.0
        return H, [1.0, 3.0], False
    if kind == "cyclic shift":
        H[i + 1, i] = 1.0
        H[0, n - 1] = 1.0
        return H, [0.0, 0.0], True
    if kind == "companion":
        H[i + 1, i] = 1.0
        H[:, n - 1] = 1.0 - np.arange(n) % 3
        return H, [0.0, 0.0, 1j, -1j], False
    if kind == "3-4-5":                  # (3, 4, 0): h00 = 0, h01 h10 + p = 3, h10 (h11 - s) = 4
        H += np.triu(np.round(3.0 * np.sin(np.arange(n * n))).reshape(n, n), 1)
        H[i + 1, i] = 1.0
        H[0, 0], H[0, 1], H[1, 0], H[1, 1], H[2, 1] = 0.0, 3.0, 1.0, 4.0, 0.0
        return H, [0.0, 0.0], False
    if kind == "1-2-2":                  # (1, 2, 2)
        H += np.triu(np.round(3.0 * np.sin(np.arange(n * n))).reshape(n, n), 1)
        H[i + 1, i] = 1.0
        H[0, 0], H[0, 1], H[1, 0], H[1, 1], H[2, 1] = 0.0, 1.0, 1.0, 2.0, 2.0
        return H, [0.0, 0.0], False
    # a first column (4, 4e, e): its squares, or only the rounding errors of
    # their sum, are below the normal range.  (With e between 1e-162 and 1e-156
    # the next columns hold nothing but entries of that size, and no reflector
    # taken from their squares is accurate.)
    e = float(kind)
    H += np.triu(np.cos(np.arange(n * n)).reshape(n, n), 1)
    H[np.arange(n), np.arange(n)] = 1.0 + np.arange(n) % 3
    H[i + 1, i] = 1.0
    H[0, 0], H[1, 0] = 2.0, e
    return H, [0.0, 0.0], False


KINDS = ["second difference", "cyclic shift", "companion", "3-4-5", "1-2-2", "1e-150", "1e-154", "1e-155",
         "1e-170", "1e-300"]


@pytest.mark.parametrize("sched", ["persistent", "sequential"])
@pytest.mark.parametrize("n,w,chain", [(5, 8, 2), (40, 16, 4), (100, 64, 16)])
@pytest.mark.parametrize("kind", KINDS)
def test_structured_sweep(gbr, kind, n, w, chain, sched):
    H, sh, exact = hessenberg(kind, n)
    Hd, Qd = gbr.to_device(H), gbr.to_device(np.eye(n))
    r = gbr.qr_sweep(Hd, Qd, sh, window=w, chain=chain, sched=sched)
    torch.cuda.synchronize()
    Hg, Qg = gbr.to_host(Hd), gbr.to_host(Qd)
    assert r.status == 0 and np.all(np.isfinite(Hg)) and np.all(np.isfinite(Qg))
    assert np.all(np.tril(Hg, -2) == 0.0)
    assert orth_err(Qg) <= 50 * n * EPS
    assert np.linalg.norm(H - Qg @ Hg @ Qg.T) <= 50 * n * EPS * np.linalg.norm(H)
    if exact:
        st, Ho, Qo = oracle.qr_sweep(H, np.eye(n), np.array(sh, complex))
        assert st == 0
        assert np.max(np.abs(Hg - Ho)) <= 50 * n * EPS and np.max(np.abs(Qg - Qo)) <= 50 * n * EPS
