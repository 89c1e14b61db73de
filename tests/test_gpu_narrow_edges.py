"""Narrow rows whose warp holds rows of very different make: windows at the
edges of the rounds the table is cleared and read in (32, 64 and 128 words;
one word wider is another kernel's), stored entries at the edges of a batch
(16 with four lanes a row, 32 with more) and none, rows of A in every slot of
a warp, and a last warp that is not full; against the CPU oracle."""
import numpy as np
import pytest

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, oracle_product, to_dev

pytestmark = pytest.mark.gpu

NBLK = 400


def _csr(rows, ncols, rng):
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    return I.Csr(len(rows), ncols, rp, np.concatenate(rows).astype(np.int32), rng.standard_normal(rp[-1]))


def _operands(n, seed):
    rng = np.random.default_rng(seed)
    a_rows, b_rows = [], []
    for i in range(n):
        width = int(rng.choice([1, 2, 31, 32, 33, 63, 64, 65, 97, 127, 128, 129]))
        lo = int(rng.integers(0, NBLK - width))
        words = np.unique(np.concatenate([[0, width - 1], rng.integers(0, width, size=4)]))
        cols = np.unique((lo + words[:, None]) * 32 + rng.integers(0, 32, size=(len(words), 4)))
        ends = cols[[0, -1]]
        first = len(b_rows)
        plen = int(rng.choice([0, 1, 3, 15, 16, 17, 31, 32, 33, 64, 65]))
        for e in range(plen):
            take = rng.choice(cols, size=int(rng.integers(0, 9)) % (len(cols) + 1), replace=False)
            b_rows.append(np.unique(np.concatenate([take, ends]) if e == 0 else take))
        a_rows.append(first + rng.permutation(plen))
    return _csr(a_rows, len(b_rows), rng), _csr(b_rows, NBLK * 32, rng)


@pytest.mark.parametrize("lanes", [4, 8, 16, 0])
@pytest.mark.parametrize("dtype,tag", [(np.float64, "f64"), (np.float32, "f32")])
@pytest.mark.parametrize("n", [1, 7, 2501])
def test_narrow_edges(cuda_lib, n, dtype, tag, lanes):
    h = sg.Handle()
    h.set_option(sg.OPT_LANES_NARROW_NUMERIC, lanes)
    h.set_option(sg.OPT_LANES_NARROW_SYMBOLIC, lanes)
    a, b = _operands(n, 11 + n)
    c = h.spgemm(to_dev(a, dtype), to_dev(b, dtype))
    h.check()
    assert_matches(c, oracle_product(a, b, dtype), tag)
