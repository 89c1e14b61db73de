"""Steps of 32 items that lie inside one row of the right-hand operand, read on
without a lookup: rows that end one before, at and one after a multiple of 32,
in the symbolic phase's block rows and in the triangle count's heavy rows."""
import numpy as np
import pytest
import torch

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, oracle_product, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens", [[31], [32], [33], [64], [1, 32, 95, 96, 97], [255, 256, 257], [320, 1], [5000]])
def test_symbolic_block_rows(cuda_lib, lens):
    rng = np.random.default_rng(sum(lens))
    nblk = 7000
    b_rows, a_rows = [], []
    for _ in range(12):
        entries = max(3, 5200 // int(np.mean(lens)))
        first = len(b_rows)
        for e in range(entries):   # a pair per entry: one column a block
            blk = np.sort(rng.choice(nblk, size=lens[e % len(lens)], replace=False))
            b_rows.append(blk * 32 + rng.integers(0, 32, size=len(blk)))
        a_rows.append(first + np.arange(entries))

    def csr(rows, ncols):
        rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
        return I.Csr(len(rows), ncols, rp, np.concatenate(rows).astype(np.int32), rng.standard_normal(rp[-1]))

    a, b = csr(a_rows, len(b_rows)), csr(b_rows, nblk * 32)
    h = sg.Handle()
    c = h.spgemm(to_dev(a), to_dev(b))
    h.check()
    assert_matches(c, oracle_product(a, b), "f64")


@pytest.mark.parametrize("n,more", [(97, 0), (300, 0), (300, 40000), (700, 900000)])
def test_clique_triangles(cuda_lib, n, more):
    """A clique of n vertices has rows of every length below n, and C(n, 3)
    triangles; with `more` isolated vertices its labels pass the bitmaps held
    by half and by one block of an SM."""
    rows = [np.delete(np.arange(n), i) for i in range(n)] + [np.zeros(0, dtype=np.int64)] * more
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    col = np.concatenate(rows[:n]).astype(np.int32)
    dev = torch.device("cuda")
    g = sg.Csr(n + more, n + more, torch.from_numpy(rp).to(dev), torch.from_numpy(col).to(dev),
               torch.ones(len(col), device=dev))
    assert sg.Handle().triangles(g) == n * (n - 1) * (n - 2) // 6
