"""What the stage kernels take from the reference matrices without reading them (CPU).

The FP32 kernel's derivative entries at P1 and P2 are compile-time constants, derived from the
Bernstein form: they have to be the FP32 values of cmcg_reference_matrices, entry for entry, with
the same zeros.  The FP64 kernel's curl, lift and inner product are the sparse Bernstein forms; the
identities are checked here against the same matrices, to the accuracy these are built to (1e-12 of
their largest entry).
"""
import itertools
import math

import numpy as np
import pytest

from paper_2106_02858_gb300 import inputs as I

FACE = ((1, 2, 3), (0, 2, 3), (0, 1, 3), (0, 1, 2))


@pytest.fixture(scope="module")
def lib():
    from paper_2106_02858_gb300 import build
    build.build()
    from paper_2106_02858_gb300 import cmcg
    return cmcg


def _bary(q):
    lat = I.node_lattice(q)
    return [tuple(b) for b in np.concatenate([q - lat.sum(1, keepdims=True), lat], axis=1)]


def _values(q):
    f = math.factorial
    b = _bary(q)
    return np.array([[f(q) / math.prod(f(int(k)) for k in a) * math.prod((x / q) ** k for x, k in zip(p, a))
                      for a in b] for p in b])


def _up(a, i, s=1):
    return tuple(x + s * (k == i) for k, x in enumerate(a))


def _bern_derivatives(q):
    b = _bary(q)
    at = {x: i for i, x in enumerate(b)}
    D = np.zeros((3, len(b), len(b)))
    low = [a for a in itertools.product(range(q), repeat=4) if sum(a) == q - 1]
    for k, a, i in itertools.product(range(3), low, range(4)):
        D[k, at[_up(a, i)], at[_up(a, k + 1)]] += a[i] + 1
        D[k, at[_up(a, i)], at[_up(a, 0)]] -= a[i] + 1
    return D


@pytest.mark.parametrize("q", [1, 2, 3])
def test_derivatives(lib, q):
    _, *D, _ = lib.cmcg_reference_matrices(q)
    B = _values(q)
    want = np.stack([B @ d @ np.linalg.inv(B) for d in _bern_derivatives(q)])
    assert np.abs(np.stack(D) - want).max() < 1e-12 * np.abs(want).max()
    if q < 3:  # whole numbers: the FP32 values are exact, zeros included
        assert np.array_equal(np.stack(D).astype(np.float32), np.round(want).astype(np.float32))
        assert np.array_equal(np.stack(D).astype(np.float32) == 0, np.round(want) == 0)


@pytest.mark.parametrize("q", [1, 2, 3])
def test_lift_and_mass(lib, q):
    M, _, _, _, L = lib.cmcg_reference_matrices(q)
    b, B = _bary(q), _values(q)
    at = {x: i for i, x in enumerate(b)}
    nfp = (q + 1) * (q + 2) // 2
    area = (math.sqrt(3) / 2, 0.5, 0.5, 0.5)
    for f in range(4):
        fb = sorted((tuple(x[v] for v in FACE[f]) for x in b if x[f] == 0),
                    key=lambda w: at[tuple(0 if v == f else w[FACE[f].index(v)] for v in range(4))])
        vol = lambda w, j: at[tuple(j if v == f else w[FACE[f].index(v)] for v in range(4))]
        fi = {w: i for i, w in enumerate(fb)}
        h = np.zeros((nfp, nfp))
        for w in fb:
            h[fi[w], fi[w]] = sum((x + 1) ** 2 for x in w)
            for i, j in itertools.permutations(range(3), 2):
                if w[j]:
                    h[fi[w], fi[_up(_up(w, i), j, -1)]] = (w[i] + 1) * w[j]
        got, level = np.zeros((len(b), nfp)), fi
        for j in range(q + 1):
            for w, r in level.items():
                got[vol(w, j)] = (-1) ** j / math.factorial(j + 1) * h[r]
            nxt = [w for w in itertools.product(range(q), repeat=3) if sum(w) == q - j - 1]
            h = np.array([sum((w[i] + 1) * h[level[_up(w, i)]] for i in range(3)) for w in nxt])
            level = {w: r for r, w in enumerate(nxt)}
        own = [vol(w, 0) for w in fb]
        want = np.linalg.solve(B, L[:, f * nfp:(f + 1) * nfp] / (2 * area[f])) @ B[np.ix_(own, own)]
        assert np.abs(got - want).max() < 1e-12 * np.abs(want).max()
    rows = [[math.prod(math.comb(x[i], g[i]) for i in range(4)) for x in b]
            for g in itertools.product(range(q + 1), repeat=4) if sum(g) <= q]
    W = np.array(rows, float)
    s = math.factorial(q) ** 2 / math.factorial(2 * q + 3)
    assert np.abs(s * W.T @ W - B.T @ M @ B).max() < 1e-12 * np.abs(M).max()
