"""Rows of C over dense windows whose row of A passes the batches after which
the windows are added up apart (1024 entries with blocks of 256 threads, 2048
with 512): entries around both and around twice both, values with infinities,
NaN and zeros of either sign; against the CPU oracle."""
import numpy as np
import pytest

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, oracle_product, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ncols", [9000, 60000])
@pytest.mark.parametrize("dtype,tag", [(np.float64, "f64"), (np.float32, "f32")])
def test_dense_folds(cuda_lib, dtype, tag, ncols):
    rng = np.random.default_rng(ncols)
    nb = 4200
    b_rows = [np.sort(rng.choice(ncols, size=int(rng.integers(1, 60)), replace=False)) for _ in range(nb)]
    b_rows[7] = np.arange(ncols)       # every window is met
    a_rows = [np.concatenate([[7], 8 + rng.choice(nb - 8, size=n - 1, replace=False)])
              for n in (600, 1023, 1024, 1025, 1536, 2047, 2048, 2049, 2560, 3072, 4096, 4097, 4190)]

    def csr(rows, n):
        rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
        return I.Csr(len(rows), n, rp, np.concatenate(rows).astype(np.int32), rng.standard_normal(rp[-1]))

    a, b = csr(a_rows, nb), csr(b_rows, ncols)
    h = sg.Handle()
    h.set_timing(True)
    c = h.spgemm(to_dev(a, dtype), to_dev(b, dtype))
    h.check()
    assert "numeric.dense" in h.timings()
    assert_matches(c, oracle_product(a, b, dtype), tag)
    # signs of zero, infinities and NaN: columns that only row 7 of B meets
    only = np.setdiff1d(np.arange(ncols), np.concatenate([b_rows[k] for k in range(8, nb)]))[:5]
    if len(only) == 5:
        b.val[b.row_ptr[7] + only] = [np.inf, -np.inf, np.nan, 0.0, -0.0]
        a.val[a.row_ptr[:-1]] = 1.0
        c = h.spgemm(to_dev(a, dtype), to_dev(b, dtype))
        h.check()
        got = c.val.cpu().numpy().reshape(len(a_rows), ncols)[:, only]
        assert np.array_equal(got, np.broadcast_to(np.array([np.inf, -np.inf, np.nan, 0.0, 0.0], dtype), got.shape),
                              equal_nan=True)
