"""The blocked back substitution at the edges of its 32-row blocks: 2x2 blocks
across a boundary, orders next to multiples of 32, vectors that need the
2^-512 scalings in several blocks (with rows above and below to rescale), real
and complex, and a leading dimension larger than n.

Against the oracle (same definition and normalization).  Well-conditioned
forms agree to rounding; in the growth patterns every sum has one dominant
term, so that vectors agree to a relative 1e-12 as well, and scaling counts
are equal.
"""
import numpy as np
import pytest

import oracle
from tests.test_gpu_eigvec import growth_matrix

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gbr():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1905_04975_gb300 as g
    g.load()
    return g


def vectors(g, S, Q=None, ld=None):
    n = S.shape[0]
    buf = torch.zeros((n, ld or n), dtype=torch.float64, device="cuda").t()[:n]
    buf.copy_(torch.from_numpy(S))
    X, ns = g.eigenvectors(buf, g.to_device(Q) if Q is not None else None, with_scalings=True)
    return X.cpu().numpy(), ns


def separated(sizes, rng):
    """Eigenvalues 1 apart with couplings 0.1: no growth, nearly normal."""
    n = int(np.sum(sizes))
    S = np.asfortranarray(np.triu(rng.standard_normal((n, n)), 1) * 0.1)
    j = 0
    for x, k in zip(rng.permutation(len(sizes)).astype(float), sizes):
        S[j, j] = x
        if k == 2:
            S[j + 1, j + 1] = x
            S[j, j + 1], S[j + 1, j] = 1.5, -0.4
        j += k
    return S


@pytest.mark.parametrize("n,sizes", [(31, 1), (32, 1), (33, 1), (64, 2), (65, "odd"), (97, "odd"), (96, "even"),
                                     (130, "mixed")])
@pytest.mark.parametrize("withq", [False, True])
def test_block_edges(gbr, n, sizes, withq):
    rng = np.random.default_rng(n)
    sz = {1: [1] * n, 2: [2] * (n // 2), "odd": [1] + [2] * (n // 2), "even": [1] + [2] * (n // 2 - 1) + [1],
          "mixed": ([1, 2, 2] * n)[:3 * (n // 5)]}[sizes]
    S = separated(sz, rng)
    n = S.shape[0]
    Q = np.asfortranarray(np.linalg.qr(rng.standard_normal((n, n)))[0]) if withq else None
    X, ns = vectors(gbr, S, Q, n + 3)
    Xo, _, _, nso = oracle.eigenvectors(S, Q)
    assert np.max(np.abs(X - Xo)) <= 1e-12 and np.array_equal(ns, nso)


@pytest.mark.parametrize("kind,n", [("gaps", 100), ("tiny pivots", 70), ("couplings", 97)])
def test_scalings_across_blocks(gbr, kind, n):
    T = np.asfortranarray(growth_matrix(kind, n))
    X, ns = vectors(gbr, T)
    Xo, _, _, nso = oracle.eigenvectors(T)
    assert np.all(np.isfinite(X)) and ns[n - 1] > 1
    assert np.array_equal(ns, nso)
    assert np.allclose(X, Xo, rtol=1e-12, atol=1e-300)


def test_complex_scalings_across_blocks(gbr):
    """2x2 blocks with couplings 2^300: a complex vector is scaled in every
    32-row block."""
    n = 80
    T = np.zeros((n, n), order="F")
    for j in range(0, n, 2):
        T[j, j] = T[j + 1, j + 1] = 1.0 + j
        T[j, j + 1], T[j + 1, j] = 1.0, -0.25
        T[j:j + 2, j + 2:] = 2.0 ** 300 * (1 + np.arange(n - j - 2) % 3)
    X, ns = vectors(gbr, T)
    Xo, _, _, nso = oracle.eigenvectors(T)
    assert np.all(np.isfinite(X)) and ns[n - 1] > 1
    assert np.array_equal(ns, nso)
    assert np.allclose(X, Xo, rtol=1e-10, atol=1e-300)
