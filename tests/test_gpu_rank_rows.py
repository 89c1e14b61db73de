"""Rows of C taken by the block-per-row dense rank accumulators, at the edges
of their ranges: column spans of one 32-column block, one run of 16 bitmap
words and the limits 2048 and 8192 blocks (and one past each), products at the
register capacity of a block (1024 and 6144) and one past it, outputs at 33,
1024, 1025, 8192 and 8193, more stored entries than a staging batch, empty
rows of B, unsorted rows of B; against the CPU oracle."""
import numpy as np
import pytest

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, oracle_product, to_dev

pytestmark = pytest.mark.gpu

# (stored entries of the row of A, entries of each of its rows of B, blocks
# of 32 columns spanned); an entry in seven meets an empty row of B
ROWS = [
    (2, 17, 2), (3, 30, 15), (3, 30, 16), (3, 30, 17), (8, 31, 500), (33, 10, 512), (40, 24, 2047), (40, 24, 2048),
    (40, 24, 2049), (130, 3, 900), (300, 2, 2048), (64, 16, 2048), (64, 17, 2048), (41, 25, 2048), (33, 32, 33),
    (200, 40, 4), (260, 30, 64), (512, 12, 8192), (513, 12, 8192), (100, 63, 3000), (128, 64, 8192), (128, 66, 8192),
    (130, 64, 8193), (1100, 9, 300), (20, 400, 1000), (700, 13, 8191),
]


def _matrices(seed, shuffle, ncols=32 * 9000):
    rng = np.random.default_rng(seed)
    a_cols, a_len, b_rows = [], [], []
    for n, blen, span in ROWS:
        base = int(rng.integers(0, 9000 - span + 1)) * 32
        first = len(b_rows)
        for e in range(n):
            if e % 7 == 3:
                b_rows.append(np.zeros(0, dtype=np.int64))
                continue
            c = base + rng.choice(32 * span, size=min(blen, 32 * span), replace=False)
            if e == 0:      # the first and the last block of the span are reached
                c = np.unique(np.concatenate([c, [base + 5, base + 32 * span - 3]]))
            b_rows.append(c if shuffle else np.sort(c))
        a_cols.append(first + np.arange(n))
        a_len.append(n)
    nb = len(b_rows)
    arp = np.concatenate([[0], np.cumsum(a_len)]).astype(np.int64)
    brp = np.concatenate([[0], np.cumsum([len(r) for r in b_rows])]).astype(np.int64)
    acol = np.concatenate(a_cols).astype(np.int32)
    bcol = np.concatenate(b_rows).astype(np.int32)
    a = I.Csr(len(ROWS), nb, arp, acol, rng.standard_normal(len(acol)))
    b = I.Csr(nb, ncols, brp, bcol, rng.standard_normal(len(bcol)))
    return a, b


@pytest.mark.parametrize("narrow", [1, 0])
@pytest.mark.parametrize("shuffle", [False, True])
@pytest.mark.parametrize("dtype,tag", [(np.float64, "f64"), (np.float32, "f32")])
def test_rank_rows_edges(cuda_lib, dtype, tag, shuffle, narrow):
    h = sg.Handle()
    h.set_option(sg.OPT_NARROW, narrow)
    a, b = _matrices(7, shuffle)
    c = h.spgemm(to_dev(a, dtype), to_dev(b, dtype))
    h.check()
    assert_matches(c, oracle_product(a, b, dtype), tag)


@pytest.mark.parametrize("nn", [33, 1024, 1025, 8192, 8193])
@pytest.mark.parametrize("dtype,tag", [(np.float64, "f64"), (np.float32, "f32")])
def test_rank_rows_outputs(cuda_lib, dtype, tag, nn):
    """One row of exactly nn outputs beside a short one: every entry reached
    once (products stored, none added), then every entry three times with
    infinities, NaN and zeros among the values (kept as the sum gives them)."""
    h = sg.Handle()
    rng = np.random.default_rng(nn)
    cols = np.sort(rng.choice(32 * 2000, size=nn, replace=False))
    for times in (1, 3):
        brp = np.concatenate([[0], np.cumsum([nn] * times + [5])]).astype(np.int64)
        bcol = np.concatenate([cols] * times + [cols[:5]]).astype(np.int32)
        b = I.Csr(times + 1, 32 * 2000, brp, bcol, rng.standard_normal(len(bcol)))
        a = I.Csr(2, times + 1, np.array([0, times, times + 1]), np.arange(times + 1, dtype=np.int32),
                  rng.standard_normal(times + 1))
        c = h.spgemm(to_dev(a, dtype), to_dev(b, dtype))
        h.check()
        assert_matches(c, oracle_product(a, b, dtype), tag)
        b.val[:6] = [np.inf, -np.inf, np.nan, 0.0, -0.0, np.inf]
        a.val[:times] = 1.0
        c = h.spgemm(to_dev(a, dtype), to_dev(b, dtype))
        h.check()
        got = c.val.double().cpu().numpy()[:6]
        want = sum(b.val[k * nn:k * nn + 6].astype(dtype).astype(np.float64) for k in range(times))
        fin = np.isfinite(want)
        assert np.array_equal(got[~fin], want[~fin], equal_nan=True)
        assert np.all(np.abs(got[fin] - want[fin]) <= 1e-5 * (1 + np.abs(want[fin])))
