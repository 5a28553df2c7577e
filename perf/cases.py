"""The work that programs have this library do, as timed cases.

Reordering a real Schur form (S, Q): the smallest forms, where a call's
latency counts; the orders of the benchmark and the tests (100, 400, 4000,
ragged ones); the largest that a program runs in one call; host buffers; a
planned batch of independent forms.  Around it the other entry points: all
eigenvectors of a form, the generalized pair (S, T), one bulge-chasing sweep.
Updates run in FP64 (the default) or, where a caller asks for it, in split
precision on the tensor cores.

Every reordering works in place, so one pass restores the form from the copy
that the program keeps and then calls the library, as a program does that
reorders the same form for several selections.

Inputs.  Strictly upper entries of a form are N(0, 1) and its eigenvalues have
the size sqrt(n) and keep apart from one another, the proportion and the
repulsion in Schur forms of dense random matrices; as more of them are real
here, their real parts are spread further, over +-4 sqrt(n).  (With
eigenvalues of size 1 under the same coupling, S would be so far from normal
that rounding alone decides its invariant subspaces.)  60% of the positions
are 1x1 blocks, the others standardized 2x2 blocks.  Q is a product of
Householder reflectors.  Pairs have S = T M on the diagonal blocks, with T's
diagonal of size sqrt(n).  A Hessenberg matrix has N(0, 1) entries above the
diagonal and the subdiagonal of a reduced dense random matrix.
"""
import math

import numpy as np
import torch

import paper_1905_04975_gb300 as gbr

F64 = torch.float64


def listed():
    return [
        # one form of a handful of eigenvalues (a pole assignment, a small
        # invariant subspace): the latency of a call
        {"name": "reorder-12", "kind": "reorder", "n": 12, "p": 0.4, "q": True, "precision": "fma",
         "window": 128, "chain": 64},
        # a small control or signal-processing form, eigenvalues only: no Q
        {"name": "reorder-100", "kind": "reorder", "n": 100, "p": 0.35, "q": False, "precision": "fma",
         "window": 128, "chain": 64},
        # the benchmark's n = 400 form at its window
        {"name": "reorder-400", "kind": "reorder", "n": 400, "p": 0.30, "q": True, "precision": "fma",
         "window": 32, "chain": 16},
        # a ragged order at the default options, from and to host arrays
        {"name": "reorder-host-1201", "kind": "host", "n": 1201, "p": 0.5, "q": True, "precision": "fma",
         "window": 128, "chain": 64},
        # the benchmark's n = 4000 form, default options
        {"name": "reorder-4000", "kind": "reorder", "n": 4000, "p": 0.35, "q": True, "precision": "fma",
         "window": 128, "chain": 64},
        # the same in split precision: chains of window tasks set the time
        {"name": "reorder-4000-split", "kind": "reorder", "n": 4000, "p": 0.35, "q": True,
         "precision": "ozaki", "window": 128, "chain": 64},
        # a large form at the default options: FP64 throughput
        {"name": "reorder-8000", "kind": "reorder", "n": 8000, "p": 0.5, "q": True, "precision": "fma",
         "window": 128, "chain": 64},
        # the largest, towards the benchmark's n = 16000, in split precision
        {"name": "reorder-12000-split", "kind": "reorder", "n": 12000, "p": 0.5, "q": True,
         "precision": "ozaki", "window": 128, "chain": 64},
        # a planned batch of independent forms of mixed orders
        {"name": "batch-512", "kind": "batch", "count": 512, "nmin": 32, "nmax": 512, "p": 0.4,
         "precision": "fma", "window": 0, "chain": 0},
        # all eigenvectors of a form, back-transformed
        {"name": "eigvec-4000", "kind": "eigvec", "n": 4000, "q": True},
        # a generalized pair with both transformations
        {"name": "pair-2000", "kind": "pair", "n": 2000, "p": 0.35, "precision": "fma", "window": 64,
         "chain": 32},
        # one bulge-chasing sweep of the Schur reduction
        {"name": "sweep-4000", "kind": "sweep", "n": 4000, "shifts": 64, "window": 64, "chain": 16},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["reorder", "reorder", "reorder", "host", "batch", "eigvec", "pair", "sweep"])
    p = round(rng.uniform(0.2, 0.6), 3)
    q = rng.random() < 0.75
    if kind == "reorder":
        n = _log(rng, 8, 8000)
        prec = rng.choice(["fma", "fma", "ozaki"])
        w, m = rng.choice([(128, 64), (128, 64), (64, 32), (96, 40)] if n > 1500 else
                          [(128, 64), (64, 32), (32, 16), (48, 20)])
        return {"kind": kind, "n": n, "p": p, "q": q, "precision": prec, "window": w, "chain": m}
    if kind == "host":
        return {"kind": kind, "n": _log(rng, 50, 3000), "p": p, "q": q, "precision": "fma", "window": 128,
                "chain": 64}
    if kind == "batch":
        return {"kind": kind, "count": _log(rng, 16, 600), "nmin": 32, "nmax": rng.choice([96, 256, 512]),
                "p": p, "precision": rng.choice(["fma", "ozaki"]), "window": 0, "chain": 0}
    if kind == "eigvec":
        return {"kind": kind, "n": _log(rng, 30, 5000), "q": q}
    if kind == "pair":
        w, m = rng.choice([(64, 32), (48, 20), (32, 12)])
        return {"kind": kind, "n": _log(rng, 30, 3000), "p": p, "precision": rng.choice(["fma", "ozaki"]),
                "window": w, "chain": m}
    return {"kind": kind, "n": _log(rng, 60, 5000), "shifts": 2 * rng.randint(2, 32), "window": 64,
            "chain": 16}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _gens(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return np.random.default_rng(seed), g


def _colmajor(n):
    return torch.empty((n, n), dtype=F64, device="cuda").t()


def _upper(n, g):
    """Strictly upper N(0, 1), column-major."""
    return torch.randn((n, n), dtype=F64, device="cuda", generator=g).tril_(-1).t()


def _block_sizes(n, rng):
    n1 = round(0.6 * n)
    n1 += (n - n1) % 2
    return rng.permutation(np.array([1] * n1 + [2] * ((n - n1) // 2)))


def _put(A, r, c, v):
    A[torch.from_numpy(r).cuda(), torch.from_numpy(c).cuda()] = torch.from_numpy(v).cuda()


def _spread(k, rng):
    """k values spread over (-4, 4), shuffled; gaps are at least 0.4 of the
    mean gap."""
    return rng.permutation(8.0 * (np.arange(k) + 0.5 + rng.uniform(-0.3, 0.3, k)) / max(k, 1) - 4.0)


def _eigen_blocks(sizes, scale, rng):
    """Diagonal, super- and subdiagonal entries of the blocks: (a, b, c) per
    position (b, c at the first row of a 2x2 block, else 0)."""
    n = int(sizes.sum())
    first = np.concatenate([[0], np.cumsum(sizes)[:-1]])
    one, two = first[sizes == 1], first[sizes == 2]
    a, b, c = np.zeros(n), np.zeros(n), np.zeros(n)
    a[one] = _spread(one.size, rng) * scale
    a[two] = a[two + 1] = _spread(two.size, rng) * scale
    # |b| and |c| apart: the standard form of a block with b = -c is any
    # rotation of it
    big, small = rng.uniform(1.0, 2.0, two.size) * scale, rng.uniform(0.1, 0.5, two.size) * scale
    sign, upper = rng.choice([-1.0, 1.0], two.size), rng.random(two.size) < 0.5
    b[two] = sign * np.where(upper, big, small)
    c[two] = -sign * np.where(upper, small, big)
    return a, b, c, two


def _form(n, rng, g, scale=None):
    """A standard real Schur form (column-major, on the GPU) and its block
    sizes."""
    sizes = _block_sizes(n, rng)
    a, b, c, two = _eigen_blocks(sizes, math.sqrt(n) if scale is None else scale, rng)
    S = _upper(n, g)
    i = np.arange(n)
    _put(S, i, i, a)
    if two.size:
        _put(S, two, two + 1, b[two])
        _put(S, two + 1, two, c[two])
    return S, sizes


def _orthogonal(n, g, k=4):
    """A product of k Householder reflectors."""
    Q = _colmajor(n)
    Q.zero_().fill_diagonal_(1.0)
    for _ in range(min(k, n)):
        v = torch.randn((n, 1), dtype=F64, device="cuda", generator=g)
        Q.addmm_(Q @ v, v.t() * (-2.0 / float((v * v).sum())))
    return Q


def _selection(sizes, p, rng):
    n = int(sizes.sum())
    first = np.concatenate([[0], np.cumsum(sizes)[:-1]])
    sel = np.zeros(n, dtype=np.int32)
    left = round(p * n)
    for b in rng.permutation(sizes.size):
        if left <= 0:
            break
        sel[first[b]:first[b] + sizes[b]] = 1
        left -= sizes[b]
    return sel


def _opts(case):
    return {"window": case["window"], "chain": case["chain"], "precision": case["precision"]}


def prepare(case, seed):
    kind = case["kind"]
    rng, g = _gens(seed)
    if kind == "batch":
        return _prepare_batch(case, rng, g)
    n = case["n"]
    if kind in ("reorder", "host", "eigvec"):
        S, sizes = _form(n, rng, g)
        Q = _orthogonal(n, g) if case["q"] else None
        st = {"kind": kind, "S0": S, "Q0": Q}
        if kind == "eigvec":
            return st
        st["sel"] = _selection(sizes, case["p"], rng)
        st["opts"] = _opts(case)
        if kind == "host":
            st["S0"] = gbr.to_host(S)
            st["Q0"] = gbr.to_host(Q) if Q is not None else None
            st["S"] = np.empty_like(st["S0"], order="F")
            st["Q"] = np.empty_like(st["Q0"], order="F") if Q is not None else None
        else:
            st["S"] = _colmajor(n)
            st["Q"] = _colmajor(n) if Q is not None else None
        return st
    if kind == "pair":
        scale = math.sqrt(n)
        sizes = _block_sizes(n, rng)
        a, b, c, two = _eigen_blocks(sizes, 1.0, rng)
        t = rng.uniform(0.5, 2.0, n) * scale
        S, T = _upper(n, g), _upper(n, g)
        i = np.arange(n)
        _put(T, i, i, t)
        _put(S, i, i, a * t)
        if two.size:
            # S_b = T_b [[a, b], [c, a]] with T_b = [[t0, t01], [0, t1]]
            t01 = rng.standard_normal(two.size)
            t0, t1, x, y, z = t[two], t[two + 1], a[two], b[two], c[two]
            _put(T, two, two + 1, t01)
            _put(S, two, two, t0 * x + t01 * z)
            _put(S, two, two + 1, t0 * y + t01 * x)
            _put(S, two + 1, two, t1 * z)
            _put(S, two + 1, two + 1, t1 * x)
        first = [S, T, _orthogonal(n, g), _orthogonal(n, g)]
        return {"kind": kind, "first": first, "work": [_colmajor(n) for _ in first],
                "sel": _selection(sizes, case["p"], rng), "opts": _opts(case)}
    # sweep
    H = torch.randn((n, n), dtype=F64, device="cuda", generator=g).tril_(0).t()
    i = np.arange(n - 1)
    _put(H, i + 1, i, np.sqrt(rng.chisquare(n - 1 - i)))
    r = math.sqrt(n)
    sh = []
    for k in range(case["shifts"] // 2):
        if k % 2 == 0:
            z = complex(rng.standard_normal() * r, rng.uniform(0.1, 1.0) * r)
            sh += [z, z.conjugate()]
        else:
            sh += [complex(x) for x in rng.standard_normal(2) * r]
    return {"kind": kind, "S0": H, "Q0": _orthogonal(n, g), "S": _colmajor(n), "Q": _colmajor(n),
            "shifts": np.array(sh), "opts": {"window": case["window"], "chain": case["chain"]}}


def _orders(case):
    """The orders of a batch's forms: the case's own, whatever the seed."""
    return np.random.default_rng(case["count"]).integers(case["nmin"], case["nmax"] + 1, case["count"])


def _prepare_batch(case, rng, g):
    """All forms of the batch in one buffer, all their Qs in another."""
    ns = _orders(case)
    off = np.concatenate([[0], np.cumsum(ns.astype(np.int64) ** 2)])
    S0 = torch.empty(int(off[-1]), dtype=F64, device="cuda")
    Q0 = torch.empty_like(S0)
    S, Q = torch.empty_like(S0), torch.empty_like(S0)
    sel = []

    def views(buf):
        return [buf[off[k]:off[k + 1]].view(n, n).t() for k, n in enumerate(ns.tolist())]

    for n, s, q in zip(ns.tolist(), views(S0), views(Q0)):
        form, sizes = _form(n, rng, g)
        s.copy_(form)
        q.copy_(_orthogonal(n, g, 1))
        sel.append(_selection(sizes, case["p"], rng))
    S.copy_(S0)
    Q.copy_(Q0)
    batch = gbr.Batch(views(S), views(Q), sel, **_opts(case))
    return {"kind": "batch", "S0": S0, "Q0": Q0, "S": S, "Q": Q, "batch": batch, "sel": sel, "ns": ns}


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind == "eigvec":
        return {"X": gbr.eigenvectors(state["S0"], state["Q0"])}
    if kind == "pair":
        for w, x in zip(state["work"], state["first"]):
            w.copy_(x)
        S, T, Q, Z = state["work"]
        r = gbr.reorder_gen(S, T, Q, Z, state["sel"], **state["opts"])
        return {"S": S, "T": T, "Q": Q, "Z": Z, "eigs": r.eigs, "m": r.m, "status": r.status}
    S, Q = state["S"], state["Q"]
    if kind == "host":
        np.copyto(S, state["S0"])
        if Q is not None:
            np.copyto(Q, state["Q0"])
        r = gbr.reorder_host(S, Q, state["sel"], **state["opts"])
    else:
        S.copy_(state["S0"])
        if Q is not None:
            Q.copy_(state["Q0"])
        if kind == "batch":
            r = state["batch"].run()
            return {"S": S, "Q": Q, "eigs": np.concatenate(r.eigs), "m": r.m, "status": r.status}
        if kind == "sweep":
            r = gbr.qr_sweep(S, Q, state["shifts"], **state["opts"])
            return {"H": S, "Q": Q, "status": r.status}
        r = gbr.reorder(S, Q, state["sel"], **state["opts"])
    out = {"S": S, "eigs": r.eigs, "m": r.m, "status": r.status}
    if Q is not None:
        out["Q"] = Q
    return out


def work(case):
    kind = case["kind"]
    if kind == "batch":
        mean2 = (case["nmin"] ** 2 + case["nmin"] * case["nmax"] + case["nmax"] ** 2) / 3
        mean3 = (case["nmin"] + case["nmax"]) * (case["nmin"] ** 2 + case["nmax"] ** 2) / 4
        p = case["p"]
        return {"bytes": case["count"] * 32 * mean2, "flops": case["count"] * 6 * p * (1 - p) * mean3}
    n = case["n"]
    if kind == "eigvec":
        # back substitution of every vector over the rows above it, and the
        # triangular product Q Y
        return {"bytes": 8 * n * n * (3 if case["q"] else 2), "flops": n ** 3 / 3 + (n ** 3 if case["q"] else 0)}
    if kind == "sweep":
        # one 3x3 reflector per bulge and row: three rows of H, three columns
        # of H and of Q
        return {"bytes": 32 * n * n, "flops": case["shifts"] / 2 * n * 2 * n * 10}
    # an adjacent swap is one rotation of two rows and two columns of S and
    # two columns of Q (12 n flops); p (1 - p) n^2 / 2 of them
    p = case["p"]
    swaps = p * (1 - p) * n * n / 2
    if kind == "pair":
        return {"bytes": 64 * n * n, "flops": swaps * 24 * n}
    q = bool(case["q"])
    return {"bytes": (32 if q else 16) * n * n, "flops": swaps * (12 if q else 6) * n}


# ---------------------------------------------------------------------------
# What has one exact value
# ---------------------------------------------------------------------------
def _first_of(S):
    """First rows of the diagonal blocks and their sizes."""
    n = S.shape[0]
    sub = np.diag(S, -1) != 0 if isinstance(S, np.ndarray) else (torch.diagonal(S, -1) != 0).cpu().numpy()
    first, size, j = [], [], 0
    while j < n:
        k = 2 if j + 1 < n and sub[j] else 1
        first.append(j)
        size.append(k)
        j += k
    return np.array(first), np.array(size)


def _order(S, sel, T=None):
    """The eigenvalues of the blocks, selected ones first, otherwise in the
    order they have (in 64 bits, from the 2x2 blocks' entries)."""
    S = torch.as_tensor(S)
    d = torch.diagonal(S).cpu().numpy()
    up, lo = torch.diagonal(S, 1).cpu().numpy(), torch.diagonal(S, -1).cpu().numpy()
    if T is not None:
        td, tu = torch.diagonal(T).cpu().numpy(), torch.diagonal(T, 1).cpu().numpy()
    ev, flag = [], []
    for j, k in zip(*_first_of(S)):
        if k == 1:
            ev.append(complex(d[j] / (td[j] if T is not None else 1.0)))
        else:
            if T is None:
                a, w = d[j], math.sqrt(-up[j] * lo[j])
            else:
                # det(S_b - x T_b) = q2 x^2 - q1 x + q0
                q2 = td[j] * td[j + 1]
                q1 = d[j] * td[j + 1] + d[j + 1] * td[j] - lo[j] * tu[j]
                q0 = d[j] * d[j + 1] - up[j] * lo[j]
                a, w = q1 / (2 * q2), math.sqrt(4 * q2 * q0 - q1 * q1) / (2 * abs(q2))
            ev += [complex(a, w), complex(a, -w)]
        flag += [bool(sel[j:j + k].any())] * k
    ev, flag = np.array(ev), np.array(flag)
    return np.concatenate([ev[flag], ev[~flag]])


def _vectors(S, Q):
    """All eigenvectors, normalized: back substitution from each eigenvalue's
    own block upwards, 64 rows at a time, then Q times them."""
    n = S.shape[0]
    first, size = _first_of(S)
    d = torch.diagonal(S).cpu().numpy()
    up, lo = torch.diagonal(S, 1).cpu().numpy(), torch.diagonal(S, -1).cpu().numpy()
    lam, start = [], []
    X = torch.zeros((n, first.size), dtype=torch.complex128, device=S.device)
    for k, (j, z) in enumerate(zip(first, size)):
        w = math.sqrt(-up[j] * lo[j]) if z == 2 else 0.0
        lam.append(complex(d[j], w))
        start.append((j, k, 1.0 + 0j))
        if z == 2:
            start.append((j + 1, k, complex(0.0, w / up[j])))
    lam = torch.tensor(lam, dtype=torch.complex128, device=S.device)
    r, c, v = zip(*start)
    X[list(r), list(c)] = torch.tensor(v, dtype=torch.complex128, device=S.device)
    own = torch.as_tensor(first, device=S.device)
    Sc = S.to(torch.complex128)
    hi = n
    bounds = set(first.tolist())
    R = -(Sc @ X)              # right-hand sides from the start vectors
    while hi > 0:
        lo_ = max(0, hi - 64)
        while lo_ not in bounds:
            lo_ -= 1
        rows = torch.arange(lo_, hi, device=S.device)
        A = Sc[lo_:hi, lo_:hi][None] - lam[:, None, None] * torch.eye(hi - lo_, dtype=torch.complex128,
                                                                      device=S.device)
        # rows at or below the eigenvalue's own block keep their start values
        keep = rows[None, :] >= own[:, None]
        eye = torch.eye(hi - lo_, dtype=torch.complex128, device=S.device)
        A = torch.where(keep[:, :, None], eye[None], A)
        rhs = torch.where(keep, torch.zeros_like(R[lo_:hi].t()), R[lo_:hi].t())
        new = torch.linalg.solve(A, rhs[:, :, None])[:, :, 0].t()
        X[lo_:hi] += new
        R[:lo_] -= Sc[:lo_, lo_:hi] @ new
        hi = lo_
    if Q is not None:
        X = Q.to(torch.complex128) @ X
    X = X / (X.real.abs() + X.imag.abs()).amax(0)
    out = torch.empty((n, n), dtype=F64, device=S.device)
    out[:, own] = X.real.contiguous()
    two = torch.as_tensor(size == 2, device=S.device)
    out[:, own[two] + 1] = X.imag[:, two].contiguous()
    return out


def _sweep(H, Q, shifts):
    """The pipelined sweep, step by step: at step t, bulge j is at t - 3 j - 1
    (-1: its introduction); the reflectors of a step, I - f v v^T with x onto
    -sign(x0) |x| e_0, are applied from the left, then from the right."""
    n, nb = H.shape[0], shifts.size // 2
    A = torch.zeros((n + 1, n + 1), dtype=F64, device=H.device)  # the last reflector has two rows
    A[:n, :n] = H
    G = torch.zeros((n, n + 1), dtype=F64, device=H.device)
    G[:, :n] = Q
    three = torch.arange(3, device=H.device)
    for t in range(n - 1 + 3 * (nb - 1)):
        j0, j1 = max(0, -((n - 2 - t) // 3)), min(nb - 1, t // 3)
        if j0 > j1:
            continue
        k = t - 1 - 3 * torch.arange(j0, j1 + 1, device=H.device)
        rows = k[:, None] + 1 + three
        x = A[rows, k.clamp(min=0)[:, None]]
        new = t == 3 * j1  # bulge j1 is introduced
        if new:
            s, p = (shifts[2 * j1] + shifts[2 * j1 + 1]).real, (shifts[2 * j1] * shifts[2 * j1 + 1]).real
            h00, h01, h10, h11, h21 = A[0, 0], A[0, 1], A[1, 0], A[1, 1], A[2, 1]
            x[-1] = torch.stack([h00 * h00 + h01 * h10 - s * h00 + p, h10 * (h00 + h11 - s), h10 * h21])
        norm = torch.linalg.vector_norm(x, dim=1)
        beta = torch.where(x[:, 0] >= 0, -norm, norm)
        v = x / (x[:, 0] - beta)[:, None]
        v[:, 0] = 1.0
        f = ((beta - x[:, 0]) / beta)[:, None]
        R = A[rows]
        A[rows] = R - (f * v)[:, :, None] * (v[:, None, :] @ R)
        k, beta = (k[:-1], beta[:-1]) if new else (k, beta)
        A[k + 1, k] = beta
        A[k + 2, k] = 0.0
        A[k + 3, k] = 0.0
        for M in (A, G):
            C = M[:, rows]
            M[:, rows] = C - (C * v).sum(-1, keepdim=True) * (f * v)
    return A[:n, :n].contiguous(), G[:, :n].contiguous()


def exact(case, seed):
    """The eigenvalues in their new order; all of an eigenvector matrix and of
    a sweep.  The other outputs are fixed up to rotations of the blocks only."""
    kind = case["kind"]
    rng, g = _gens(seed)
    if kind == "sweep":
        st = prepare(case, seed)
        H, Q = _sweep(st["S0"], st["Q0"], st["shifts"])
        return {"H": H, "Q": Q, "status": None}
    if kind == "eigvec":
        S, _ = _form(case["n"], rng, g)
        return {"X": _vectors(S, _orthogonal(case["n"], g) if case["q"] else None)}
    if kind == "batch":
        eigs = []
        for n in _orders(case).tolist():
            S, sizes = _form(n, rng, g)
            _orthogonal(n, g, 1)
            eigs.append(_order(S, _selection(sizes, case["p"], rng)))
        return {"S": None, "Q": None, "eigs": np.concatenate(eigs), "m": None, "status": None}
    if kind == "pair":
        st = prepare(case, seed)
        S, T = st["first"][:2]
        return {"S": None, "T": None, "Q": None, "Z": None, "eigs": _order(S, st["sel"], T), "m": None,
                "status": None}
    S, sizes = _form(case["n"], rng, g)
    if case["q"]:
        _orthogonal(case["n"], g)
    return {"S": None, "Q": None, "eigs": _order(S, _selection(sizes, case["p"], rng)), "m": None,
            "status": None}
