"""Single swaps of close eigenvalues are as exact as those of separated ones.

A form of decoupled quads: 16 to 64 pairs of neighbouring blocks, coupled only
within the pair, the lower block of each selected.  Its window's first step
swaps every pair; the exchanges between pairs that follow have a zero coupling,
so that their Sylvester solutions are zero and their transformations exact
permutations.  Q then holds each pair's own transformation, and the part of
Q^T D Q (Q^T D Z) that the swap has to make vanish is evaluated in extended
precision.

Against the same statistic at a separation of 1: only the Sylvester solution
sees the separation, the reflectors and products after it do not, and a
backward stable solution leaves a residual of a rounding or two at any
separation.  Twice the largest error at separation 1 allows for the solution's
part being as large as all others together, and for the spread of a maximum.
"""
import numpy as np
import pytest

from tests.helpers import orth_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps
LD = np.longdouble


@pytest.fixture(scope="module")
def gbr():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1905_04975_gb300 as g
    g.load()
    return g


def quads(rng, count, pairs, size, sep):
    """count x pairs diagonal blocks D = [[A, C], [0, B]] of two size x size
    blocks: eigenvalues sep apart on the real axis, the same imaginary part,
    couplings of the size of the separation."""
    k = 2 * size
    D = np.zeros((count, pairs, k, k))
    x = rng.standard_normal((count, pairs))
    y = x + sep * rng.choice([-1.0, 1.0], (count, pairs))
    b, c = rng.uniform(1.0, 2.0, (count, pairs)), -rng.uniform(0.2, 0.5, (count, pairs))
    for o, v in ((0, x), (size, y)):
        for i in range(size):
            D[..., o + i, o + i] = v
        if size == 2:
            D[..., o, o + 1], D[..., o + 1, o] = b, c
    D[..., :size, size:] = sep * rng.standard_normal((count, pairs, size, size))
    return D


def assemble(D):
    """Block-diagonal matrices (count x n x n) of the quads."""
    count, pairs, k, _ = D.shape
    S = np.zeros((count, pairs * k, pairs * k))
    for p in range(pairs):
        S[:, p * k:(p + 1) * k, p * k:(p + 1) * k] = D[:, p]
    return S


def pair_factors(Q, pairs, size):
    """The pairs' own transformations, count x pairs x k x k: rows of the pair,
    columns of its swapped (leading) and its other block."""
    k, m = 2 * size, pairs * size
    out = np.empty((Q.shape[0], pairs, k, k))
    for p in range(pairs):
        cols = [p * size + i for i in range(size)] + [m + p * size + i for i in range(size)]
        out[:, p] = Q[:, p * k:(p + 1) * k][:, :, cols]
    return out


def vanishing(D, Q, Z, size):
    """max of the block that must vanish, in eps times the largest entry of D."""
    P = np.einsum("...ab,...ac,...cd->...bd", Q.astype(LD), D.astype(LD), Z.astype(LD), optimize=True)
    low = np.abs(P[..., size:, :size]).max(axis=(-1, -2))
    return (low / np.abs(D).max(axis=(-1, -2)) / EPS).astype(float)


def window_errors(g, sep, seed, size, count=512):
    """Errors of count x 32 (64) swaps of size x size blocks."""
    pairs = 128 // (2 * size)
    D = quads(np.random.default_rng(seed), count, pairs, size, sep)
    S = torch.from_numpy(assemble(D)).cuda()
    n = S.shape[1]
    # column-major views: the transpose of a row-major transpose
    Sd = [s.t().contiguous().t() for s in S]
    Qd = [torch.eye(n, dtype=torch.float64, device="cuda").t() for _ in range(count)]
    sel = np.tile(np.repeat([0, 1], size), pairs).astype(np.int32)
    r = g.Batch(Sd, Qd, [sel] * count, window=128, chain=64).run()
    assert np.all(r.status == 0)
    Q = torch.stack(Qd).cpu().numpy()
    assert max(orth_err(q) for q in Q[::64]) <= 50 * n * EPS
    F = pair_factors(Q, pairs, size)
    return vanishing(D, F, F, size)


@pytest.mark.parametrize("size", [1, 2])
def test_window_swaps(gbr, size):
    ref = window_errors(gbr, 1.0, 1, size)
    for i, sep in enumerate([1e-2, 1e-3, 1e-4, 3e-5, 1e-5, 3e-6, 1e-6, 1e-7]):
        e = window_errors(gbr, sep, 10 + i, size)
        assert e.max() <= 2.0 * ref.max(), sep
        assert e.mean() <= 1.25 * ref.mean(), sep


def gen_errors(g, sep, seed, size, count=60):
    """The same for pairs (S, T), with T's diagonal in [1, 2]; every swap has
    to be accepted, as a backward stable one is."""
    pairs = 64 // (2 * size)
    rng = np.random.default_rng(seed)
    M = quads(rng, count, pairs, size, sep)
    k = 2 * size
    B = sep * np.triu(rng.standard_normal((count, pairs, k, k)), 1)
    for i in range(k):
        B[..., i, i] = rng.uniform(1.0, 2.0, (count, pairs))
    A = np.zeros_like(M)
    for o in (0, size):  # diagonal blocks T_b M_b, so that S T^-1 has M's eigenvalues
        A[..., o:o + size, o:o + size] = B[..., o:o + size, o:o + size] @ M[..., o:o + size, o:o + size]
    A[..., :size, size:] = M[..., :size, size:]
    S, T = assemble(A), assemble(B)
    n = S.shape[1]
    sel = np.tile(np.repeat([0, 1], size), pairs).astype(np.int32)
    Qs, Zs, rejected = [], [], 0
    for s, t in zip(S, T):
        d = [g.to_device(x) for x in (s, t, np.eye(n), np.eye(n))]
        rejected += g.reorder_gen(*d, sel, window=64, chain=32).status
        Qs.append(g.to_host(d[2]))
        Zs.append(g.to_host(d[3]))
    assert rejected == 0, (sep, rejected)
    Q, Z = pair_factors(np.array(Qs), pairs, size), pair_factors(np.array(Zs), pairs, size)
    return np.maximum(vanishing(A, Q, Z, size), vanishing(B, Q, Z, size))


@pytest.mark.parametrize("size", [1, 2])
def test_pair_swaps(gbr, size):
    ref = gen_errors(gbr, 1.0, 1, size, 120)
    for i, sep in enumerate([1e-2, 1e-3, 1e-4, 3e-5, 1e-5, 3e-6, 1e-6, 1e-7]):
        e = gen_errors(gbr, sep, 10 + i, size, 120)
        assert e.max() <= 2.0 * ref.max(), sep
        assert e.mean() <= 1.25 * ref.mean(), sep
