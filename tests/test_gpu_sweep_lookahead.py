"""Sweeps at the edges of the window task's look-ahead: a bulge reaching the
last rows (its reflector shrinks to two rows, then it leaves the chain), a new
bulge introduced at every third step, windows so short that the look-ahead runs
for one or two steps, the widest window with as many bulges as it holds, and
matrices whose squares leave the normal range.

Against the oracle, element by element: rounding differences grow along the
chase with the number of shifts (1e-8 is the bound of the other sweep tests).
"""
import numpy as np
import pytest

import oracle
import schur_inputs as si
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


def check(g, H, Q, sh, **kw):
    n = H.shape[0]
    Hd, Qd = g.to_device(H), g.to_device(Q)
    g.qr_sweep(Hd, Qd, sh, **kw)
    torch.cuda.synchronize()
    Hg, Qg = g.to_host(Hd), g.to_host(Qd)
    st, Ho, Qo = oracle.qr_sweep(H, Q, sh)
    assert st == 0 and np.all(np.tril(Hg, -2) == 0.0)
    assert orth_err(Qg) <= 50 * n * EPS
    A = Q @ H @ Q.T
    assert np.linalg.norm(A - Qg @ Hg @ Qg.T) <= 50 * n * EPS * np.linalg.norm(A)
    assert np.linalg.norm(Hg - Ho) <= 1e-8 * np.linalg.norm(H)
    assert np.max(np.abs(Qg - Qo)) <= 1e-8


@pytest.mark.parametrize("n", [3, 4, 5, 6, 8, 9, 12, 13, 25])
@pytest.mark.parametrize("w,chain", [(8, 2), (12, 4), (96, 32)])
def test_ends_of_the_matrix(gbr, n, w, chain):
    H, Q, sh = si.hessenberg_problem(n, 40 + n, nshifts=4, reflectors=2)
    check(gbr, H, Q, sh, window=w, chain=chain)


@pytest.mark.parametrize("n,ns,w,chain", [(60, 16, 48, 16), (150, 32, 96, 32), (200, 12, 18, 6), (97, 20, 64, 20)])
def test_many_bulges(gbr, n, ns, w, chain):
    H, Q, sh = si.hessenberg_problem(n, n + ns, nshifts=ns, reflectors=4)
    check(gbr, H, Q, sh, window=w, chain=chain)


@pytest.mark.parametrize("e", [-470, 470])
def test_scaled_rows(gbr, e):
    """The rows and columns from 20 on scaled by 2^e: the chase there works on
    reflectors whose sums of squares lie next to the ends of the normal range.
    (The whole matrix cannot be: the introduction multiplies entries.)"""
    n = 60
    H, Q, sh = si.hessenberg_problem(n, 9, nshifts=4, reflectors=4)
    H[20:, 20:] *= 2.0 ** e
    Hd, Qd = gbr.to_device(H), gbr.to_device(Q)
    gbr.qr_sweep(Hd, Qd, sh, window=24, chain=4)
    torch.cuda.synchronize()
    Hg, Qg = gbr.to_host(Hd), gbr.to_host(Qd)
    assert np.all(np.isfinite(Hg)) and np.all(np.tril(Hg, -2) == 0.0)
    assert orth_err(Qg) <= 50 * n * EPS
    m = np.max(np.abs(H))
    assert np.linalg.norm(Q @ (H / m) @ Q.T - Qg @ (Hg / m) @ Qg.T) <= 50 * n * EPS * np.linalg.norm(H / m)
