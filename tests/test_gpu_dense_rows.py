"""Rows of C taken by the windows of the dense accumulator (sorted rows of B,
many products over their span): one window exactly full, one column more, and
several windows in FP32 and FP64; parts of rows of B of 1, 63, 64, 65, 128 and
more entries (whole strips and flat ends); more stored entries than a staging
batch of 512; entries whose every product is -0.0, infinities and NaN; against
the CPU oracle."""
import numpy as np
import pytest

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, oracle_product, to_dev

pytestmark = pytest.mark.gpu


def _csr(rows, ncols, rng):
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    col = np.concatenate(rows).astype(np.int32)
    return I.Csr(len(rows), ncols, rp, col, rng.standard_normal(len(col)))


def _operands(ncols, seed):
    """B: rows of every strip remainder over all columns, some empty, some
    within one window; A: rows of 60, 513 and 1300 entries and short ones."""
    rng = np.random.default_rng(seed)
    lens = [1, 63, 64, 65, 127, 128, 129, 300, 1000, 0, 40, 2000]
    b_rows = []
    for k in range(1400):
        n = min(lens[k % len(lens)], ncols)
        if k % 5 == 4:      # a dense run of columns
            c0 = int(rng.integers(0, ncols - n + 1))
            b_rows.append(np.arange(c0, c0 + n))
        else:
            b_rows.append(np.sort(rng.choice(ncols, size=n, replace=False)))
    b_rows[3] = np.array([0, ncols - 1])
    a_rows = [np.sort(rng.choice(1400, size=n, replace=False)) for n in (60, 513, 1300, 3, 200, 511, 512, 1, 1400)]
    return _csr(a_rows, 1400, rng), _csr(b_rows, ncols, rng)


@pytest.mark.parametrize("ncols", [2000, 10240, 12288, 12289, 22528, 24577, 70001])
@pytest.mark.parametrize("dtype,tag", [(np.float64, "f64"), (np.float32, "f32")])
def test_dense_rows_windows(cuda_lib, dtype, tag, ncols):
    h = sg.Handle()
    h.set_timing(True)
    a, b = _operands(ncols, ncols)
    c = h.spgemm(to_dev(a, dtype), to_dev(b, dtype))
    h.check()
    assert "numeric.dense" in h.timings()
    assert_matches(c, oracle_product(a, b, dtype), tag)


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_dense_rows_special_values(cuda_lib, dtype):
    """Entries whose products are all -0.0 stay in the pattern (as zeros),
    sums that cancel stay, infinities and NaN come out as the sum gives them."""
    h = sg.Handle()
    n, times = 9000, 4
    cols = np.arange(0, 2 * n, 2)
    b = I.Csr(times, 2 * n, np.arange(times + 1, dtype=np.int64) * n, np.tile(cols, times).astype(np.int32),
              np.tile(np.arange(n) % 7 - 3.0, times))
    b.val[:n:3] = 0.0
    for k in range(1, times):
        b.val[k * n:(k + 1) * n:3] = 0.0
    a = I.Csr(1, times, np.array([0, times]), np.arange(times, dtype=np.int32), np.array([-1.0, -2.0, -1.0, -4.0]))
    b.val[[1, 4]] = [np.inf, np.nan]
    b.val[n + 1] = -np.inf
    c = h.spgemm(to_dev(a, dtype), to_dev(b, dtype))
    h.check()
    assert np.array_equal(c.col.cpu().numpy(), cols)
    got = c.val.double().cpu().numpy()
    want = sum(a.val[k] * b.val[k * n:(k + 1) * n] for k in range(times))
    assert np.array_equal(got, want, equal_nan=True)      # small whole numbers: exact
    assert not np.signbit(got[::3]).any()                  # a zero sum is +0.0, as from a zeroed accumulator
    # a sum that cancels exactly
    a2 = I.Csr(1, 2, np.array([0, 2]), np.array([0, 1], dtype=np.int32), np.array([1.0, -1.0]))
    b2 = I.Csr(2, 2 * n, np.array([0, n, 2 * n]), np.tile(cols, 2).astype(np.int32), np.tile(np.arange(n) + 1.0, 2))
    c = h.spgemm(to_dev(a2, dtype), to_dev(b2, dtype))
    h.check()
    assert c.nnz == n and not c.val.any()
