"""Rows of C of at most 512 products taken by the kernel with two levels of
bitmaps: products at the edges of a step (32), of a warp's slots (256, 257)
and of the class (512, 513), spans at the edges of a word of the first bitmap
(32 and 33 blocks), of a round of its scan (1024 and 1025) and of the class
(8192 and 8193), non-empty blocks at the edges of a round of the second one
(128, 129), more stored entries than are staged at a time (32), empty rows of
B, unsorted rows of B, alone and together with longer rows, few and many;
against the CPU oracle."""
import numpy as np
import pytest

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, oracle_product, to_dev

pytestmark = pytest.mark.gpu

NBLK = 8400


def _csr(rows, ncols, rng):
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    return I.Csr(len(rows), ncols, rp, np.concatenate(rows).astype(np.int32), rng.standard_normal(rp[-1]))


def _operands(shuffle, longer, times, seed):
    rng = np.random.default_rng(seed)
    a_rows, b_rows = [], []

    def row(products, span, entries, blocks=None):
        """A row of A of `entries` entries (one in nine meeting an empty row
        of B) and `products` products over `span` blocks, both ends met."""
        base = int(rng.integers(0, NBLK - span + 1)) * 32
        cols = base + rng.permutation(32 * span)[:max(2, (2 * products) // 3)]
        if blocks:
            cols = base + 32 * rng.permutation(span)[:blocks] + rng.integers(0, 32, size=blocks)
        cols[:2] = base + 5, base + 32 * span - 3
        cols = np.unique(cols)
        full = [e for e in range(entries) if e % 9 != 4]
        cut = np.sort(rng.choice(np.arange(1, products), size=len(full) - 1, replace=False)) if len(full) > 1 else []
        lens = np.diff(np.concatenate([[0], cut, [products]])).astype(int)
        first, left = len(b_rows), rng.permutation(cols)
        for e in range(entries):
            n = lens[full.index(e)] if e in full else 0
            take = left[:n]
            left = left[n:]
            if len(take) < n:
                rest = np.setdiff1d(cols, take)
                take = np.concatenate([take, rng.choice(rest, size=min(n - len(take), len(rest)), replace=False)])
            b_rows.append(rng.permutation(take) if shuffle else np.sort(take))
        a_rows.append(first + np.arange(entries))

    for span in (4, 32, 33, 150, 1024, 1025, 2048, 2049, 8191, 8192, 8193):
        for products in (34, 64, 255, 256, 257, 320, 511, 512, 513):
            for entries in (6, 32, 33):
                row(products, span, entries)
        row(400, span, 130)
    for blocks in (127, 128, 129, 256, 257, 400):
        row(450, 2000, 20, blocks)
    if longer:
        for _ in range(5):
            row(900, 1500, 40)
            row(4000, 3000, 70)
    a_rows = a_rows * times
    order = rng.permutation(len(a_rows))
    return _csr([a_rows[k] for k in order], len(b_rows), rng), _csr(b_rows, NBLK * 32, rng)


@pytest.mark.parametrize("times", [1, 70])
@pytest.mark.parametrize("longer", [False, True])
@pytest.mark.parametrize("shuffle", [False, True])
@pytest.mark.parametrize("dtype,tag,native", [(np.float64, "f64", 1), (np.float32, "f32", 1), (np.float64, "f64", 0)])
def test_short_rows(cuda_lib, dtype, tag, native, shuffle, longer, times):
    h = sg.Handle()
    h.set_timing(True)
    h.set_option(sg.OPT_F64_NATIVE, native)
    a, b = _operands(shuffle, longer, times, 3 + longer)
    c = h.spgemm(to_dev(a, dtype), to_dev(b, dtype))
    h.check()
    assert_matches(c, oracle_product(a, b, dtype), tag)
    if native:
        assert "numeric.rank_short" in h.timings()


@pytest.mark.parametrize("rows", [300, 21000])
@pytest.mark.parametrize("dtype,tag", [(np.float64, "f64"), (np.float32, "f32")])
def test_short_rows_with_longer_ones(cuda_lib, dtype, tag, rows):
    """Spans within 2048 blocks: few short rows share the longer rows' launch,
    many have their own."""
    rng = np.random.default_rng(rows)
    n = 3000
    b = _csr([np.sort(rng.choice(n, size=int(rng.integers(4, 33)), replace=False)) for _ in range(n)], n, rng)
    a = _csr([rng.choice(n, size=int(rng.integers(4, 33)), replace=False) for _ in range(rows)], n, rng)
    h = sg.Handle()
    h.set_timing(True)
    c = h.spgemm(to_dev(a, dtype), to_dev(b, dtype))
    h.check()
    assert_matches(c, oracle_product(a, b, dtype), tag)
    assert ("numeric.rank_short" in h.timings()) == (rows == 21000)


def test_short_rows_special_values(cuda_lib):
    """Infinities, NaN and zeros met once and twice; the sum keeps them."""
    rng = np.random.default_rng(9)
    cols = np.sort(rng.choice(32 * 3000, size=200, replace=False))
    for dtype in (np.float32, np.float64):
        b = _csr([cols, cols, cols[:6]], 32 * 3000, rng)
        b.val[:6] = [np.inf, -np.inf, np.nan, 0.0, -0.0, np.inf]
        b.val[200:206] = [-np.inf, 1.0, 2.0, 0.0, -0.0, np.inf]
        a = I.Csr(2, 3, np.array([0, 2, 3]), np.arange(3, dtype=np.int32), np.ones(3))
        c = sg.Handle().spgemm(to_dev(a, dtype), to_dev(b, dtype))
        got = c.val.double().cpu().numpy()
        with np.errstate(invalid="ignore"):
            want = b.val[:6] + b.val[200:206]
        assert np.array_equal(got[:6], want, equal_nan=True)
        assert np.array_equal(np.signbit(got[3:5]), np.signbit(want[3:5]))
