"""Triangles of hubs joined to one another that share more than 2^20 leaves:
rows of L too long for a batch's columns to be numbered in an int, looked up row
by row, with the bitmap in shared memory (n below 1,572,864) and in global
memory.  Every common leaf closes one triangle with each pair of hubs and every
three hubs close one, so the counts have a closed form."""
import math

import numpy as np
import pytest

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LEAVES = 1_100_000


@pytest.mark.parametrize("hubs", [2, 3])
@pytest.mark.parametrize("n", [LEAVES + 7, 1_700_000])
def test_joined_hubs(cuda_lib, n, hubs):
    """Hub j has j leaves of its own beside the common ones, so the hubs'
    labels are in order: hub j is the highest-labelled vertex of LEAVES * j
    triangles with a leaf and of C(j, 2) with two hubs."""
    hub = np.arange(hubs, dtype=np.int64) * (n // hubs)
    rest = np.setdiff1d(np.arange(n, dtype=np.int64), hub)
    own = [rest[LEAVES + j * (j - 1) // 2:][:j] for j in range(hubs)]
    x, y = np.triu_indices(hubs, 1)
    a = np.concatenate([np.repeat(hub, LEAVES), hub[x]] + [np.full(j, hub[j]) for j in range(hubs)])
    b = np.concatenate([np.tile(rest[:LEAVES], hubs), hub[y]] + own)
    g = I._coo_to_csr(n, np.concatenate([a, b]), np.concatenate([b, a]))
    h = sg.Handle()
    G = sg.Csr.from_host(g, "cuda", np.float32)
    want = np.zeros(n, dtype=np.int64)
    want[hub] = [LEAVES * j + math.comb(j, 2) for j in range(hubs)]
    for _ in range(5):
        total, perm, vc = h.triangles(G, labels=True)
        assert np.all(np.diff(perm.cpu().numpy()[hub]) > 0)
        assert total == LEAVES * math.comb(hubs, 2) + math.comb(hubs, 3)
        assert np.array_equal(vc.cpu().numpy(), want)
