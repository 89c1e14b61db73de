"""Rows of C with more than 8192 outputs over sorted rows of B: dense windows or
windows walked by cursors, by what either costs in the type.  Rows of which both
types, one type only and neither take dense windows, all in one product, enough
of them that the cursors are used and few enough that they are not; rows over rows
of B of two entries, where the other choice is the rank accumulators; values and
patterns against the CPU oracle, the kernels from the rows they were launched on."""
import numpy as np
import pytest

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, oracle_product, to_dev

pytestmark = pytest.mark.gpu

# entries of a row of A, entries of its rows of B, columns they lie in
SPARSE = (100, 100, 1_000_000)
DENSE = (200, 100, 100_000)
FP32 = (2000, 40, 1_000_000)     # sparse, but a sum may have thousands of terms, which FP32 folds
FP64 = (25, 500, 400_000)


def _product(groups, rows, rng):
    """A and B: `rows` rows of A a group, each group on rows of B of its own."""
    ncols = max(g[2] for g in groups)
    b_rows, a_rows = [], []
    for alen, per, width in groups:
        k0 = len(b_rows)
        b_rows += [np.unique(rng.integers(0, width, size=per)) for _ in range(3 * alen)]
        a_rows += [k0 + np.sort(rng.choice(3 * alen, size=alen, replace=False)) for _ in range(rows)]

    def csr(r, n):
        rp = np.concatenate([[0], np.cumsum([len(x) for x in r])]).astype(np.int64)
        return I.Csr(len(r), n, rp, np.concatenate(r).astype(np.int32), rng.standard_normal(rp[-1]))

    return csr(a_rows, len(b_rows)), csr(b_rows, ncols)


def _run(a, b, dtype, tag):
    h = sg.Handle()
    h.set_timing(True)
    c = h.spgemm(to_dev(a, dtype), to_dev(b, dtype))
    h.check()
    assert_matches(c, oracle_product(a, b, dtype), tag)
    return {k: (v[0], v[1]) for k, v in h.timings().items() if k.startswith("numeric.")}


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("dtype,tag", [(np.float64, "f64"), (np.float32, "f32")])
def test_lists(cuda_lib, dtype, tag):
    rows = _sms() + 5     # two lists of them are more than two for each SM
    t = _run(*_product([SPARSE, DENSE, FP32, FP64], rows, np.random.default_rng(1)), dtype, tag)
    assert t["numeric.dense"][1] == 2 * rows
    # FP32: the rows for FP64 alone lie apart from those for neither
    assert t["numeric.bin6_window"] == ((1 if tag == "f64" else 2), 2 * rows)


@pytest.mark.parametrize("dtype,tag", [(np.float64, "f64"), (np.float32, "f32")])
def test_few_rows(cuda_lib, dtype, tag):
    rows = _sms() // 2
    t = _run(*_product([SPARSE, DENSE, FP32, FP64], rows, np.random.default_rng(2)), dtype, tag)
    assert t["numeric.dense"][1] == 4 * rows and "numeric.bin6_window" not in t


@pytest.mark.parametrize("group", [SPARSE, DENSE, FP32, FP64])
@pytest.mark.parametrize("dtype,tag", [(np.float64, "f64"), (np.float32, "f32")])
def test_one_list(cuda_lib, dtype, tag, group):
    t = _run(*_product([group], 2 * _sms() + 1, np.random.default_rng(3)), dtype, tag)
    dense = group is DENSE or group is (FP64 if tag == "f64" else FP32)
    assert ("numeric.dense" in t, "numeric.bin6_window" in t) == (dense, not dense), t


@pytest.mark.parametrize("alen,width,kernel", [(4000, 40_000, "numeric.rank_long"), (3080, 9_000, "numeric.dense"),
                                               (4000, 20_000, "numeric.dense"), (4000, 60_000, "numeric.rank_long")])
@pytest.mark.parametrize("dtype,tag", [(np.float64, "f64"), (np.float32, "f32")])
def test_short_rows_of_b(cuda_lib, dtype, tag, alen, width, kernel):
    """Rows of C of 4097 to 8192 outputs, two products an entry of A."""
    t = _run(*_product([(alen, 2, width)], 40, np.random.default_rng(4)), dtype, tag)
    assert set(t) - {"numeric.dense_split"} == {kernel}, t
