"""Unsorted rows of B whose entries jump between blocks: a row of 32 to 128
blocks then has more (block, mask) pairs than a window has words, and stays a
narrow row's; against the CPU oracle."""
import numpy as np
import pytest

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, oracle_product, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lanes", [0, 4, 16])
@pytest.mark.parametrize("dtype,tag", [(np.float64, "f64"), (np.float32, "f32")])
def test_more_pairs_than_words(cuda_lib, dtype, tag, lanes):
    rng = np.random.default_rng(4)
    rows = []
    for span in (1, 2, 33, 128):
        for cols in (20, 32, 129, 200, 900):
            c = np.sort(rng.choice(32 * span, size=min(cols, 32 * span), replace=False)) + 32 * int(rng.integers(0, 50))
            rows.append(rng.permutation(c))
            # few distinct columns a block, met in turns
            rows.append(rng.permutation(np.unique(c - c % 32)))
    col = np.concatenate(rows).astype(np.int32)
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    b = I.Csr(len(rows), 32 * 200, rp, col, rng.standard_normal(len(col)))
    a = I.Csr(len(rows), len(rows), np.arange(len(rows) + 1), np.arange(len(rows), dtype=np.int32),
              rng.standard_normal(len(rows)))
    h = sg.Handle()
    h.set_option(sg.OPT_LANES_NARROW_NUMERIC, lanes)
    h.set_option(sg.OPT_LANES_NARROW_SYMBOLIC, lanes)
    c = h.spgemm(to_dev(a, dtype), to_dev(b, dtype))
    h.check()
    assert_matches(c, oracle_product(a, b, dtype), tag)
