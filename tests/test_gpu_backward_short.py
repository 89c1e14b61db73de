"""Gradients where the rows have few products in the mean (one or two steps of 32
at a time in place of four): rows of 31 to 300 products, and the same with 40 and
with 5000 rows of 0 to 6 products among them; rows of B in any order, empty ones
among them; against the oracle."""
import numpy as np
import pytest
import torch

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_grads_match, host_csr, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("short,mean", [(0, (64, 1000)), (40, (32, 64)), (5000, (0, 32))])
@pytest.mark.parametrize("dtype,tol", [(np.float64, 1e-12), (np.float32, 1e-5)])
def test_gradients(cuda_lib, dtype, tol, short, mean):
    rng = np.random.default_rng(short + 1)
    ncols, a_rows, b_rows = 3000, [], []
    for n in [31, 32, 33, 63, 64, 65, 96, 97, 128, 129, 160, 300] * 4:
        first = len(b_rows)
        cut = np.sort(rng.choice(n + 1, size=5))
        for x in np.diff(np.concatenate([[0], cut, [n]])):
            b_rows.append(rng.choice(ncols, size=x, replace=False))
        a_rows.append(first + rng.permutation(len(b_rows) - first))
    for _ in range(short):
        first = len(b_rows)
        for x in rng.integers(0, 3, size=rng.integers(0, 4)):
            b_rows.append(rng.choice(ncols, size=x, replace=False))
        a_rows.append(first + rng.permutation(len(b_rows) - first))
    order = rng.permutation(len(a_rows))

    def csr(r, m):
        rp = np.concatenate([[0], np.cumsum([len(x) for x in r])]).astype(np.int64)
        return I.Csr(len(r), m, rp, np.concatenate(r).astype(np.int32), rng.standard_normal(rp[-1]).astype(dtype).astype(np.float64))

    a, b = csr([a_rows[x] for x in order], len(b_rows)), csr(b_rows, ncols)
    assert mean[0] < a.nnz * b.nnz / (a.nrows * b.nrows) <= mean[1]
    h = sg.Handle()
    A, B = to_dev(a, dtype), to_dev(b, dtype)
    c = h.spgemm(A, B)
    dc = torch.linspace(-1, 1, c.nnz, dtype=c.val.dtype, device="cuda")
    for need_a, need_b in ((True, True), (True, False), (False, True)):
        da, db = h.backward(A, B, c, dc, need_a, need_b)
        h.check()
        assert (da is None) == (not need_a) and (db is None) == (not need_b)
    da, db = h.backward(A, B, c, dc)
    h.check()
    hc = host_csr(c)
    assert_grads_match(a, b, hc.row_ptr, hc.col, dc.cpu().numpy(), da.cpu().numpy(), db.cpu().numpy(), tol)
