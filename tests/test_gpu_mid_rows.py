"""Rows of C of 513 to 1024 products over more than 2048 blocks of 32 columns:
products at 512, 513, 1023, 1024 and 1025, spans at 2048, 2049, 8192 and 8193
blocks, more stored entries than are staged at a time, empty rows of B,
unsorted rows of B; against the CPU oracle."""
import numpy as np
import pytest

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, oracle_product, to_dev

pytestmark = pytest.mark.gpu

NBLK = 8400


@pytest.mark.parametrize("shuffle", [False, True])
@pytest.mark.parametrize("dtype,tag,native", [(np.float64, "f64", 1), (np.float32, "f32", 1), (np.float64, "f64", 0)])
def test_mid_rows(cuda_lib, dtype, tag, native, shuffle):
    rng = np.random.default_rng(17)
    a_rows, b_rows = [], []
    for span in (2048, 2049, 5000, 8192, 8193):
        for products in (512, 513, 1023, 1024, 1025):
            for entries in (4, 33, 100):
                base = int(rng.integers(0, NBLK - span + 1)) * 32
                cols = np.unique(np.concatenate([[base + 1, base + 32 * span - 1],
                                                 base + rng.choice(32 * span, size=(3 * products) // 4, replace=False)]))
                lens = np.full(entries, products // entries)
                lens[:products % entries] += 1
                first = len(b_rows)
                left = rng.permutation(cols)
                for n in lens:
                    take, left = left[:n], left[n:]
                    if len(take) < n:
                        take = np.concatenate([take, rng.choice(np.setdiff1d(cols, take), size=n - len(take), replace=False)])
                    b_rows.append(rng.permutation(take) if shuffle else np.sort(take))
                b_rows.append(np.zeros(0, dtype=np.int64))
                a_rows.append(first + rng.permutation(entries + 1))

    def csr(rows, ncols):
        rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
        return I.Csr(len(rows), ncols, rp, np.concatenate(rows).astype(np.int32), rng.standard_normal(rp[-1]))

    a, b = csr(a_rows, len(b_rows)), csr(b_rows, NBLK * 32)
    h = sg.Handle()
    h.set_timing(True)
    h.set_option(sg.OPT_F64_NATIVE, native)
    c = h.spgemm(to_dev(a, dtype), to_dev(b, dtype))
    h.check()
    assert_matches(c, oracle_product(a, b, dtype), tag)
    if native:
        assert "numeric.rank_mid" in h.timings()
