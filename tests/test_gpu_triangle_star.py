"""Triangle count of stars: one row of L with millions of entries and nothing to
look up, whose work must grow with its entries, not with their square; and stars
whose hubs take turns on a block (a row's bits cleared when the next row's are
set), against the closed form."""
import math

import numpy as np
import pytest

import paper_1804_00695_gb300 as sg

pytestmark = pytest.mark.gpu


def _csr(n, a, b):
    import torch
    r, c = torch.cat([a, b]), torch.cat([b, a])
    key = torch.sort(r * n + c)[0]
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(key // n, minlength=n), 0, out=rp[1:])
    return sg.Csr(n, n, rp, (key % n).int(), torch.ones(len(key), device="cuda"))


def _ms(h, g, want):
    import torch
    best = math.inf
    for _ in range(4):
        e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        e0.record()
        assert h.triangles(g) == want
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best


def test_star_work_is_linear(cuda_lib):
    """Four times the leaves: four times the work, sixteen if every task of a
    row set all its bits again.  Both bitmaps are in global memory."""
    import torch
    h = sg.Handle()

    def star(n):
        hub = torch.full((n,), n // 2, device="cuda")
        leaf = torch.cat([torch.arange(n // 2, device="cuda"), torch.arange(n // 2 + 1, n + 1, device="cuda")])
        return _csr(n + 1, hub, leaf)

    few, many = _ms(h, star(2_000_000), 0), _ms(h, star(8_000_000), 0)
    assert many < 8 * few, (few, many)


@pytest.mark.parametrize("n", [300_000, 900_000, 1_700_000])
def test_rows_taken_in_turn(cuda_lib, n):
    """600 hubs of 300 to 1500 leaves in rings of 3, each ring on leaves of its
    own: a block meets tasks of many rows, one after another.  Every leaf of a
    ring closes three triangles (its three hubs two by two), the hubs one."""
    import torch
    rng = np.random.default_rng(n)
    ids = rng.permutation(n)
    hubs, leaves = ids[:600].reshape(200, 3), ids[600:]
    sizes = rng.integers(300, 1500, size=200)
    sizes = np.minimum(sizes, (len(leaves) - 1) // 200)
    at = np.concatenate([[0], np.cumsum(sizes)])
    a, b = [], []
    for r in range(200):
        own = leaves[at[r]:at[r + 1]]
        for j in range(3):
            a += [np.full(len(own), hubs[r, j]), hubs[r, j:j + 1]]
            b += [own, hubs[r, (j + 1) % 3:(j + 1) % 3 + 1]]
    t = [torch.from_numpy(np.concatenate(x).astype(np.int64)).cuda() for x in (a, b)]
    g = _csr(n, *t)
    h = sg.Handle()
    for _ in range(2):
        total, perm, vc = h.triangles(g, labels=True)
        assert total == 3 * int(sizes.sum()) + 200
        # the highest-labelled vertex of every one of them is a hub: the ring's
        # top hub closes two a leaf and the hubs' own, the middle one one a leaf
        vc, perm = vc.cpu().numpy(), perm.cpu().numpy()
        want = np.zeros(n, dtype=np.int64)
        order = np.argsort(perm[hubs], axis=1)
        for r in range(200):
            want[hubs[r, order[r, 2]]] = 2 * sizes[r] + 1
            want[hubs[r, order[r, 1]]] = sizes[r]
        assert np.array_equal(vc, want)
