"""Swaps of the pair window task at the edges of their ranges: many swaps of
one kind in a step, S and T of very different scales, a T with a zero diagonal
entry (an infinite eigenvalue) and eigenvalues so close that the FP32-seeded
generalized Sylvester solution has to give way to the elimination.

Checked is what any backward stable swap satisfies: the generalized
eigenvalues in the expected order, exact structure, Q and Z orthogonal and
(S, T) = Q (S', T') Z^T within 50 n eps (an accepted swap has a backward error
of at most 20 eps of its blocks, and they add up like a random walk over the
about n swaps that touch an entry).
"""
import numpy as np
import pytest

from tests.helpers import EPS, blocks, orth_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gbr():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1905_04975_gb300 as g
    g.load()
    return g


def pair(sizes, rng, gap, coupling):
    """A pair whose blocks' eigenvalues are gap apart (real parts), shuffled;
    T's diagonal between 1 and 2."""
    n = int(np.sum(sizes))
    S = np.asfortranarray(np.triu(rng.standard_normal((n, n)), 1) * coupling)
    T = np.asfortranarray(np.triu(rng.standard_normal((n, n)), 1) * coupling)
    T[np.diag_indices(n)] = rng.uniform(1.0, 2.0, n)
    lam = rng.permutation(len(sizes)) * gap
    j, ev = 0, []
    for x, k in zip(lam, sizes):
        if k == 1:
            S[j, j] = x * T[j, j]
            ev.append(complex(x))
        else:
            S[j:j + 2, j:j + 2] = T[j:j + 2, j:j + 2] @ np.array([[x, 1.5], [-0.4, x]])
            ev += [complex(x, np.sqrt(0.6)), complex(x, -np.sqrt(0.6))]
        j += k
    return S, T, np.array(ev)


def run_and_check(g, S, T, sel, want, w, tol, sched="persistent"):
    n = S.shape[0]
    d = [g.to_device(x) for x in (S, T, np.eye(n), np.eye(n))]
    r = g.reorder_gen(*d, sel, window=w, chain=w // 2, sched=sched)
    torch.cuda.synchronize()
    S1, T1, Q, Z = (g.to_host(x) for x in d)
    assert r.status == 0 and r.m == int(np.sum(sel))
    flag = sel.astype(bool)
    assert np.max(np.abs(r.eigs - np.concatenate([want[flag], want[~flag]]))) <= tol
    assert np.all(np.tril(S1, -2) == 0.0) and np.all(np.tril(T1, -1) == 0.0)
    assert sum(k for _, k in blocks(S1)) == n
    assert orth_err(Q) <= 50 * n * EPS and orth_err(Z) <= 50 * n * EPS
    for X, Y in ((S, S1), (T, T1)):
        scale = np.max(np.abs(X))
        d = (X - Q @ Y @ Z.T) / scale
        assert np.linalg.norm(d) <= 50 * n * EPS * np.linalg.norm(X / scale)


@pytest.mark.parametrize("kinds", ["2x2 only", "1x1 only", "1x1 above 2x2", "2x2 above 1x1", "mixed"])
@pytest.mark.parametrize("n,w", [(64, 64), (66, 64), (100, 32)])
def test_many_swaps_of_a_kind(gbr, kinds, n, w):
    rng = np.random.default_rng(n + w)
    sizes = {"2x2 only": [2] * (n // 2), "1x1 only": [1] * n, "1x1 above 2x2": [1, 2] * (n // 3),
             "2x2 above 1x1": [2, 1] * (n // 3), "mixed": list(rng.integers(1, 3, 2 * n // 3))}[kinds]
    S, T, ev = pair(sizes, rng, 1.0, 0.3)
    sel = np.repeat(np.arange(len(sizes)) % 2, sizes).astype(np.int32)
    run_and_check(gbr, S, T, sel, ev, w, 1e-10 * len(sizes))


@pytest.mark.parametrize("s,t", [(0, -400), (400, 0), (-400, -400), (300, -300)])
def test_scaled_pairs(gbr, s, t):
    """Powers of two on S and T scale the eigenvalues and nothing else.  With
    both at 2^-400 the discriminants of the 2x2 blocks underflow, and the
    validation refuses the pair."""
    rng = np.random.default_rng(5)
    sizes = list(rng.integers(1, 3, 30))
    S, T, ev = pair(sizes, rng, 1.0, 0.3)
    sel = (rng.random(len(sizes)) < 0.4).repeat(sizes).astype(np.int32)
    f = 2.0 ** (s - t)
    if s == t == -400:
        with pytest.raises(gbr.GbrError) as e:
            run_and_check(gbr, np.asfortranarray(S * 2.0 ** s), np.asfortranarray(T * 2.0 ** t), sel, ev, 64, 1.0)
        assert e.value.status == -2
        return
    run_and_check(gbr, np.asfortranarray(S * 2.0 ** s), np.asfortranarray(T * 2.0 ** t), sel, ev * f, 64,
                  1e-10 * len(sizes) * f)


def test_infinite_eigenvalue(gbr):
    rng = np.random.default_rng(6)
    sizes = [1] * 24
    S, T, ev = pair(sizes, rng, 1.0, 0.3)
    S[10, 10], T[10, 10] = 1.0, 0.0
    sel = np.zeros(24, np.int32)
    sel[[10, 15, 20]] = 1
    d = [gbr.to_device(x) for x in (S, T, np.eye(24), np.eye(24))]
    r = gbr.reorder_gen(*d, sel, window=32, chain=12)
    S1, T1, Q, Z = (gbr.to_host(x) for x in d)
    assert r.status == 0 and abs(r.eigs[0]) > 1e12
    assert np.max(np.abs(r.eigs[1:3] - ev[[15, 20]])) <= 1e-9
    for X, Y in ((S, S1), (T, T1)):
        assert np.linalg.norm(X - Q @ Y @ Z.T) <= 50 * 24 * EPS * np.linalg.norm(X)


@pytest.mark.parametrize("sched", ["persistent", "sequential"])
@pytest.mark.parametrize("gap", [1e-2, 1e-4, 1e-6])
def test_close_eigenvalues(gbr, gap, sched):
    """Couplings of the size of the gap keep the swaps well enough conditioned
    to be accepted."""
    rng = np.random.default_rng(13)
    sizes = [2, 2, 1, 2, 1, 2, 2, 1] * 4
    S, T, ev = pair(sizes, rng, gap, gap)
    sel = np.repeat(np.arange(len(sizes)) % 2 == 1, sizes).astype(np.int32)
    run_and_check(gbr, S, T, sel, ev, 64, 1e-9, sched)
