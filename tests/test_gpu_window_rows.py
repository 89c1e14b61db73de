"""Narrow rows of more than 32 outputs, and narrow rows too few to fill the
chip, taken by the window kernels with an accumulator per subgroup: outputs at
33, 255, 256 and 257, words at 32 and 33, products around the change from a
warp to a block, more stored entries than a batch (64 for a warp, 256 for a
block), rows of B of 1 to 70 entries, empty ones and unsorted ones, alone and
mixed with rows of other kernels; against the CPU oracle."""
import numpy as np
import pytest

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, oracle_product, to_dev

pytestmark = pytest.mark.gpu

NCOLS = 32 * 700


def _csr(rows, ncols, rng):
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    return I.Csr(len(rows), ncols, rp, np.concatenate(rows).astype(np.int32), rng.standard_normal(rp[-1]))


def _operands(shuffle, seed, wide=False):
    rng = np.random.default_rng(seed)
    a_rows, b_rows = [], []

    def row(nn, words, blens):
        """A row of nn outputs in `words` words of a window of at most 128,
        its rows of B drawn from them (the first ones cover all)."""
        blk = int(rng.integers(0, 700 - 128)) + np.sort(rng.choice(128, size=words, replace=False))
        cols = np.unique(np.concatenate([blk[np.arange(nn) % words] * 32 + np.arange(nn) // words]))
        assert len(cols) == nn
        first = len(b_rows)
        left = cols.copy()
        for n in blens:
            take = left[:n] if len(left) else rng.choice(cols, size=min(n, nn), replace=False)
            left = left[n:]
            b_rows.append(rng.permutation(take) if shuffle else np.sort(take))
        assert not len(left)
        a_rows.append(first + np.arange(len(blens)))

    for nn, words in ((33, 2), (33, 33), (64, 32), (64, 33), (200, 7), (255, 20), (256, 32), (256, 8), (257, 9), (300, 33)):
        row(nn, words, [40] * 9)
        row(nn, words, [70, 0, 1, 17] + [16] * 20)
        row(nn, words, [15] * 65)
        row(nn, words, [33] * 124)           # 4092 products
        row(nn, words, [32] * 128)           # 4096
        row(nn, words, [64] * 300 + [3])
    for nn in (1, 5, 31, 32):
        row(nn, min(nn, 6), [nn] * 3)
        row(nn, min(nn, 6), [nn] + [max(1, nn // 2)] * 500)
    if wide:
        for _ in range(30):
            first = len(b_rows)
            b_rows.extend(np.sort(rng.choice(NCOLS, size=60, replace=False)) for _ in range(12))
            a_rows.append(first + np.arange(12))
    order = rng.permutation(len(a_rows))
    return _csr([a_rows[k] for k in order], len(b_rows), rng), _csr(b_rows, NCOLS, rng)


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("shuffle", [False, True])
@pytest.mark.parametrize("dtype,tag,native", [(np.float64, "f64", 1), (np.float32, "f32", 1), (np.float64, "f64", 0)])
def test_window_rows(cuda_lib, dtype, tag, native, shuffle, wide):
    h = sg.Handle()
    h.set_timing(True)
    h.set_option(sg.OPT_F64_NATIVE, native)
    a, b = _operands(shuffle, 5 + wide, wide)
    c = h.spgemm(to_dev(a, dtype), to_dev(b, dtype))
    h.check()
    assert_matches(c, oracle_product(a, b, dtype), tag)
    if native:
        assert {"numeric.window_warp", "numeric.window_block", "numeric.narrow"} <= set(h.timings())


@pytest.mark.parametrize("n", [4, 13, 30])
@pytest.mark.parametrize("lanes", [0, 4])
def test_few_narrow_rows(cuda_lib, n, lanes):
    """Every row narrow: the lanes per row follow the number of rows (a few
    rows: a warp or a block each), and the forced choice gives the same."""
    h = sg.Handle()
    h.set_option(sg.OPT_LANES_NARROW_NUMERIC, lanes)
    h.set_option(sg.OPT_LANES_NARROW_SYMBOLIC, lanes)
    a, p, r = I.galerkin_problem(n)
    for x, y in ((a, p), (r, a)):
        c = h.spgemm(to_dev(x), to_dev(y))
        h.check()
        assert_matches(c, oracle_product(x, y), "f64")
