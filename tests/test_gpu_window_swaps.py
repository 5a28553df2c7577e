"""Swap transforms of the window task at the edges of their ranges: many swaps
of one kind in a step (several groups of a warp's swaps), entries whose squares
leave the normal range, decoupled blocks, and eigenvalues so close that the
FP32-seeded Sylvester solution has to give way to the elimination.

Compared with the oracle where the subspaces are well separated, otherwise by
what any backward stable swap satisfies: the eigenvalue order, the standard
form, Q orthogonal and A = Q S Q^T within 50 n eps (an accepted swap has a
backward error of at most 10 eps max|D|, and they add up like a random walk
over the about n swaps that touch an entry).
"""
import numpy as np
import pytest

import oracle
from tests.helpers import EPS, block_eigs, expected_order, is_standard, orth_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gbr():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1905_04975_gb300 as g
    g.load()
    return g


def form(sizes, rng, gap, coupling):
    """A standard form whose blocks' eigenvalues are gap apart on the real
    axis, shuffled."""
    n = int(np.sum(sizes))
    S = np.asfortranarray(np.triu(rng.standard_normal((n, n)), 1) * coupling)
    a = rng.permutation(len(sizes)) * gap
    j = 0
    for x, k in zip(a, sizes):
        S[j, j] = x
        if k == 2:
            S[j + 1, j + 1] = x
            S[j, j + 1], S[j + 1, j] = rng.uniform(1.0, 2.0), -rng.uniform(0.2, 0.5)
        j += k
    return S


def run(g, S, sel, w, sched="persistent"):
    Sd, Qd = g.to_device(S), g.to_device(np.eye(S.shape[0]))
    r = g.reorder(Sd, Qd, sel, window=w, chain=w // 2, sched=sched)
    torch.cuda.synchronize()
    return r, g.to_host(Sd), g.to_host(Qd)


def check(S, sel, r, Sg, Qg):
    n, scale = S.shape[0], np.max(np.abs(S))
    want, m = expected_order(S, sel)
    assert r.status == 0 and r.m == m and is_standard(Sg)
    assert np.max(np.abs(r.eigs - block_eigs(Sg))) <= 1e-14 * scale
    assert np.max(np.abs(block_eigs(Sg) - want)) <= 1e-10 * scale
    assert orth_err(Qg) <= 50 * n * EPS
    d = (S - Qg @ Sg @ Qg.T) / scale
    assert np.linalg.norm(d) <= 50 * n * EPS * np.linalg.norm(S / scale)


@pytest.mark.parametrize("kinds", ["2x2 only", "1x1 only", "1x1 above 2x2", "2x2 above 1x1", "mixed"])
@pytest.mark.parametrize("n,w", [(128, 128), (66, 128), (130, 64), (200, 200)])
def test_many_swaps_of_a_kind(gbr, kinds, n, w):
    """Interleaved selection: about n / 4 swaps in a step (with 2x2 blocks
    more than the two, with mixed ones more than the eight of a group)."""
    rng = np.random.default_rng(n + w)
    k = n // 2
    sizes = {"2x2 only": [2] * k, "1x1 only": [1] * n, "1x1 above 2x2": [1, 2] * (n // 3),
             "2x2 above 1x1": [2, 1] * (n // 3), "mixed": list(rng.integers(1, 3, 2 * n // 3))}[kinds]
    S = form(sizes, rng, 1.0, 0.3)
    sel = np.repeat(np.arange(len(sizes)) % 2, sizes).astype(np.int32)
    r, Sg, Qg = run(gbr, S, sel, w)
    check(S, sel, r, Sg, Qg)
    ref = oracle.reorder(S, np.eye(S.shape[0]), sel)
    assert ref["status"] == 0
    m = r.m
    P, R = Qg[:, :m], ref["Q"][:, :m]
    assert np.linalg.norm(P - R @ (R.T @ P), 2) <= 1e-10


@pytest.mark.parametrize("scale", [2.0 ** -480, 2.0 ** -400, 2.0 ** 400, 2.0 ** 480])
def test_scaled_forms(gbr, scale):
    """Scaling by a power of two changes no decision: the transformations of
    the scaled form are those of the form itself, up to the rotations whose
    squares need their own scaling (a few roundings)."""
    rng = np.random.default_rng(7)
    sizes = list(rng.integers(1, 3, 50))
    S = form(sizes, rng, 1.0, 0.5)
    sel = (rng.random(len(sizes)) < 0.4).repeat(sizes).astype(np.int32)
    _, S1, Q1 = run(gbr, S, sel, 128)
    r, Sg, Qg = run(gbr, np.asfortranarray(S * scale), sel, 128)
    check(S * scale, sel, r, Sg, Qg)
    n = S.shape[0]
    assert np.linalg.norm(Qg - Q1) <= 50 * n * EPS * np.sqrt(n)
    assert np.linalg.norm(Sg / scale - S1) <= 50 * n * EPS * np.linalg.norm(S)


@pytest.mark.parametrize("coupling", [0.0, 2.0 ** -300])
def test_decoupled_blocks(gbr, coupling):
    rng = np.random.default_rng(11)
    sizes = [2, 1, 2, 2, 1, 1, 2, 1] * 4
    S = form(sizes, rng, 1.0, coupling)
    sel = np.repeat(np.arange(len(sizes)) % 3 == 1, sizes).astype(np.int32)
    r, Sg, Qg = run(gbr, S, sel, 128)
    check(S, sel, r, Sg, Qg)


@pytest.mark.parametrize("sched", ["persistent", "sequential"])
@pytest.mark.parametrize("gap", [1e-2, 1e-4, 1e-6])
def test_close_eigenvalues(gbr, gap, sched):
    """Normal couplings of the size of the gap keep the swaps well enough
    conditioned to be accepted; the separation of the blocks goes from where
    the FP32-seeded solution converges to where it cannot."""
    rng = np.random.default_rng(13)
    sizes = [2, 2, 1, 2, 1, 2, 2, 1] * 4
    S = form(sizes, rng, gap, gap)
    j = 0
    for k in sizes:  # the same imaginary part for every pair
        if k == 2:
            S[j, j + 1], S[j + 1, j] = 1.5, -0.4
        j += k
    sel = np.repeat(np.arange(len(sizes)) % 2 == 1, sizes).astype(np.int32)
    r, Sg, Qg = run(gbr, S, sel, 128, sched)
    check(S, sel, r, Sg, Qg)
