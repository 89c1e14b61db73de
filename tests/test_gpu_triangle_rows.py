"""Triangle counting at the edges of its kernels: rows of L of 64 and 65 entries
(a warp or a block), of 256, 257 and 512 and 513 (tasks of a block), vertices of
more than 1024 neighbours (their row of L by a block), vertices of degree 0 to 2,
and graphs whose bitmap takes blocks of 512 or 1024 threads; counts and
per-vertex counts against the oracle."""
import math

import numpy as np
import pytest

import oracle
import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _graph(n, a, b):
    keep = a != b
    a, b = a[keep], b[keep]
    return I._coo_to_csr(n, np.concatenate([a, b]), np.concatenate([b, a]))


def _clique(ids):
    k = len(ids)
    x, y = np.triu_indices(k, 1)
    return ids[x], ids[y]


def _check(g):
    h = sg.Handle()
    G = sg.Csr.from_host(g, "cuda", np.float32)
    total, perm, vc = h.triangles(G, labels=True)
    perm = perm.cpu().numpy()
    assert np.array_equal(np.sort(perm), np.arange(g.nrows))
    deg = np.diff(g.row_ptr)
    assert np.all(np.diff(deg[np.argsort(perm)]) >= 0)
    want, per = oracle.triangles(g, perm)
    assert total == want and np.array_equal(vc.cpu().numpy(), per)
    assert h.triangles(G) == total
    return total


@pytest.mark.parametrize("k", [3, 65, 66, 257, 258, 513, 514, 1026])
def test_cliques(cuda_lib, k):
    """A clique spread over the ids, with pendant and isolated vertices: its
    rows of L have 0 to k - 1 entries."""
    n = 4 * k + 7
    ids = (np.arange(k, dtype=np.int64) * 3 + 2)
    a, b = _clique(ids)
    pend = np.arange(n - 6, n - 1, dtype=np.int64)
    g = _graph(n, np.concatenate([a, pend]), np.concatenate([b, ids[np.arange(5) % k]]))
    assert _check(g) == math.comb(k, 3)


@pytest.mark.parametrize("n", [5000, 700000, 900000])
def test_hubs(cuda_lib, n):
    """Hubs of several thousand neighbours joined to one another, over few and
    many columns (bitmaps of 157, 21,875 and 28,125 words)."""
    rng = np.random.default_rng(n)
    hubs = rng.choice(n, size=30, replace=False).astype(np.int64)
    a, b = _clique(hubs)
    others = rng.choice(n, size=4000, replace=False).astype(np.int64)
    src = np.repeat(hubs, 3000)
    dst = rng.choice(others, size=len(src))
    x, y = rng.choice(others, size=20000), rng.choice(others, size=20000)
    g = _graph(n, np.concatenate([a, src, x]), np.concatenate([b, dst, y]))
    assert _check(g) > math.comb(30, 3)
