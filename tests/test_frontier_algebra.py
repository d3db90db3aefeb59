"""The wedge form of the frontier engine, checked on the CPU with the oracle's
field multiply: eliminating the source's row from the label space and taking
the wedge product of the other vertices' rows gives the permanent the sieve
points sum to, whatever the pivot; a slip in the elimination does not."""
import itertools

import numpy as np
import pytest

import oracle


@pytest.fixture(scope="module", autouse=True)
def _lib():
    oracle.build()


def _perm(rows):
    """Permanent by its definition: every bijection of rows and labels."""
    k, acc = len(rows), 0
    for p in itertools.permutations(range(k)):
        t = 1
        for i, j in enumerate(p):
            t = oracle.gf_mul(t, rows[i][j])
        acc ^= t
    return acc


def _wedge(rows, slip=False):
    """z_{s,p} times the wedge of the other rows over the labels without p."""
    k, zs = len(rows), rows[0]
    p = next((j for j, v in enumerate(zs) if v), None)
    if p is None:
        return 0
    inv = oracle.gf_inv(zs[p])
    rho = [oracle.gf_mul(v, inv) for v in zs]
    labels = [j for j in range(k) if j != p]
    state = {frozenset(): zs[p]}
    for z in rows[1:]:
        zr = [z[j] ^ (0 if slip else oracle.gf_mul(z[p], rho[j])) for j in labels]
        new = {}
        for S, v in state.items():
            for j in range(k - 1):
                if j not in S:
                    T = S | {j}
                    new[T] = new.get(T, 0) ^ oracle.gf_mul(zr[j], v)
        state = new
    return state[frozenset(range(k - 1))]


@pytest.mark.parametrize("k", [2, 3, 4, 5, 6])
@pytest.mark.parametrize("zeros", [0, 1, 2])
def test_wedge_is_the_permanent(k, zeros):
    rng = np.random.default_rng(100 * k + zeros)
    for _ in range(4):
        rows = [[int(x) for x in r] for r in rng.integers(1, 2**63, (k, k))]
        for j in range(min(zeros, k)):
            rows[0][j] = 0
        want = _perm(rows)
        assert _wedge(rows) == want
        if k > 2 and zeros == 0:
            assert _wedge(rows, slip=True) != want


def test_a_repeated_vertex_vanishes():
    rng = np.random.default_rng(7)
    rows = [[int(x) for x in r] for r in rng.integers(1, 2**63, (5, 5))]
    for a, b in ((0, 3), (1, 4)):
        rep = [list(r) for r in rows]
        rep[b] = list(rep[a])
        assert _wedge(rep) == 0 == _perm(rep)
