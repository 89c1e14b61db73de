"""FP32 rows over dense windows whose entries are sums of many terms: blocks of 256
threads (8000 columns, folded every 1024 entries of the row of A) and of 512 (60,000
columns, every 2048), entries around one, two and three folds; values of every
sign and kind in columns of their own; and a sum that only folds keep."""
import numpy as np
import pytest

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, oracle_product, to_dev

pytestmark = pytest.mark.gpu

FOLD = {8000: 1024, 60000: 2048}


def _csr(rows, ncols, vals):
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    return I.Csr(len(rows), ncols, rp, np.concatenate(rows).astype(np.int32), vals(rp[-1]))


def _run(a, b, dtype):
    h = sg.Handle()
    h.set_timing(True)
    c = h.spgemm(to_dev(a, dtype), to_dev(b, dtype))
    h.check()
    assert "numeric.dense" in h.timings()
    return c


@pytest.mark.parametrize("ncols", [8000, 60000])
@pytest.mark.parametrize("dtype,tag", [(np.float64, "f64"), (np.float32, "f32")])
def test_edges(cuda_lib, dtype, tag, ncols):
    rng = np.random.default_rng(ncols + 1)
    nb, kinds = 4200, 5                       # the first columns: row 0 of B alone
    b_rows = [kinds + np.sort(rng.choice(ncols - kinds, size=int(rng.integers(1, 60)), replace=False)) for _ in range(nb)]
    b_rows[0] = np.arange(ncols)              # every window is met
    a_rows = [np.concatenate([[0], 1 + np.sort(rng.choice(nb - 1, size=n - 1, replace=False))])
              for n in (900, 1023, 1024, 1025, 1026, 1536, 2047, 2048, 2049, 2050, 3071, 3072, 3073, 4095, 4096, 4097, 4190)]
    a, b = _csr(a_rows, nb, rng.standard_normal), _csr(b_rows, ncols, rng.standard_normal)
    assert_matches(_run(a, b, dtype), oracle_product(a, b, dtype), tag)
    b.val[:kinds] = [np.inf, -np.inf, np.nan, 0.0, -0.0]
    a.val[a.row_ptr[:-1]] = 1.0
    c = _run(a, b, dtype)
    got = c.val.cpu().numpy().reshape(len(a_rows), ncols)[:, :kinds]
    want = np.broadcast_to(np.array([np.inf, -np.inf, np.nan, 0.0, 0.0], dtype), got.shape)
    assert np.array_equal(got, want, equal_nan=True)
    assert not np.signbit(got[:, 3:]).any()   # a sum of zeros starts from +0


@pytest.mark.parametrize("ncols", [8000, 60000])
def test_small_terms_are_kept(cuda_lib, ncols):
    """Column 0 sums 2^24 and then 1/2 for every other entry of the row of A: in
    FP32 2^24 + 1/2 rounds to 2^24, so one chain of additions loses all that come
    after the first block-wide batch of entries, while folds add up the terms of
    every fold among themselves, exactly, and lose at most those beside 2^24 and
    one rounding (to a multiple of 2) a fold."""
    rng = np.random.default_rng(ncols)
    n = 20000
    b_rows = [np.concatenate([[0], 1 + np.sort(rng.choice(ncols - 1, size=3, replace=False))]) for _ in range(n)]
    a = _csr([np.arange(n)] * 3, n, np.ones)
    b = _csr(b_rows, ncols, np.ones)
    b.val[b.row_ptr[:-1]] = 0.5
    b.val[0] = 2.0 ** 24
    c = _run(a, b, np.float32)
    rp = c.row_ptr.cpu().numpy()[:-1]
    assert np.array_equal(c.col.cpu().numpy()[rp], np.zeros(3))
    lost = 2.0 ** 24 + 0.5 * (n - 1) - c.val.cpu().numpy()[rp].astype(np.float64)
    limit = 0.5 * FOLD[ncols] + (n // FOLD[ncols] + 1)
    assert limit < 0.5 * (n - 512)            # what one chain would lose at least
    assert np.all(np.abs(lost) <= limit), lost
