"""The first numeric call after a symbolic one under stream capture: the row lists
are then made when the graph runs, so a call on the stream itself before the graph
has run makes its own, as one after it does.  Narrow rows with empty rows between
them (listed since the others lie between), and rows of every other kind."""
import numpy as np
import pytest
import torch

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, oracle_product, to_dev

pytestmark = pytest.mark.gpu


def _narrow():
    """Banded, every third row of A empty."""
    n = 900
    rows = np.repeat(np.arange(n), 3)
    cols = np.minimum(rows + np.tile([0, 2, 5], n), n - 1)
    keep = rows % 3 != 1
    key = np.unique(rows[keep] * n + cols[keep])
    rp = np.concatenate([[0], np.cumsum(np.bincount(key // n, minlength=n))]).astype(np.int64)
    a = I.Csr(n, n, rp, (key % n).astype(np.int32), np.linspace(-1, 1, len(key)))
    return a, I.laplace2d_5pt(30)


def _mixed():
    a = I.random_csr(500, 600, 0.05, 5)
    return a, I.random_csr(600, 30000, 0.002, 6)


@pytest.mark.parametrize("make", [_narrow, _mixed])
@pytest.mark.parametrize("dtype,tag", [(np.float64, "f64"), (np.float32, "f32")])
def test_capture_first(cuda_lib, make, dtype, tag):
    a, b = make()
    A, B = to_dev(a, dtype), to_dev(b, dtype)
    ref = oracle_product(a, b, dtype)
    assert_matches(sg.Handle().spgemm(A, B), ref, tag)   # loads every kernel
    h = sg.Handle()
    rp, nnz = h.symbolic(A, B)
    c = sg.Csr(A.nrows, B.ncols, rp, torch.zeros(nnz, dtype=torch.int32, device="cuda"), torch.zeros_like(A.val[:1]).repeat(nnz))
    torch.cuda.synchronize()
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s):
            h.numeric_into(A, B, c)

    def run(f):
        c.col.zero_()
        c.val.zero_()
        torch.cuda.synchronize()
        f()
        torch.cuda.synchronize()
        h.check()
        assert_matches(c, ref, tag)

    run(lambda: h.numeric_into(A, B, c))   # before the graph has run
    run(g.replay)
    run(lambda: h.numeric_into(A, B, c))
    h.set_option(sg.OPT_SMALL_CAP, 16)     # lists from another class on
    run(lambda: h.numeric_into(A, B, c))
    run(g.replay)
    run(lambda: h.numeric_into(A, B, c))
    h.set_option(sg.OPT_SMALL_CAP, 32)
    run(lambda: h.numeric_into(A, B, c))
    rp2, nnz2 = h.symbolic(A, B)           # a new symbolic call: lists on the stream again
    c = h.numeric(A, B, rp2, nnz2)
    h.check()
    assert_matches(c, ref, tag)
