"""Gradients at the edges of the row kernel's steps: rows of 0, 1, 2, 31, 32,
33, 127, 128, 129 and 257 products, of 1, 2, 1023, 1024 and 1025 outputs, more
stored entries than are staged at a time (32), empty rows of B between the
others, unsorted rows of B; against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


def _csr(rows, ncols, rng):
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    return I.Csr(len(rows), ncols, rp, np.concatenate(rows).astype(np.int32), rng.standard_normal(rp[-1]))


def _operands(seed):
    rng = np.random.default_rng(seed)
    ncols, a_rows, b_rows = 4000, [], []

    def row(lens, cols):
        first = len(b_rows)
        for n in lens:
            b_rows.append(rng.choice(cols, size=min(n, len(cols)), replace=False))
        a_rows.append(first + rng.permutation(len(lens)))

    for outputs in (1, 2, 40, 1023, 1024, 1025):
        cols = rng.choice(ncols, size=outputs, replace=False)
        row([outputs], cols)                                   # every output is met
        row([0, outputs, 0, 0, outputs], cols)
        row([outputs] + [min(outputs, 3)] * 40, cols)
    for products in (0, 1, 2, 31, 32, 33, 127, 128, 129, 257):
        cols = rng.choice(ncols, size=300, replace=False)
        row([products], cols)
        row([1] * products, cols)
        row([0] * 5 + [products // 2, 0, products - products // 2] + [0] * 30, cols)
    return _csr(a_rows, len(b_rows), rng), _csr(b_rows, ncols, rng)


@pytest.mark.parametrize("dtype,tag", [(np.float64, "f64"), (np.float32, "f32")])
def test_backward_steps(cuda_lib, dtype, tag):
    a, b = _operands(21)
    h = sg.Handle()
    A, B = to_dev(a, dtype), to_dev(b, dtype)
    C = h.spgemm(A, B)
    dc = np.random.default_rng(5).standard_normal(C.nnz).astype(dtype)
    da, db = h.backward(A, B, C, torch.from_numpy(dc).cuda())
    h.check()
    ra64 = I.Csr(a.nrows, a.ncols, a.row_ptr, a.col, a.val.astype(dtype).astype(np.float64))
    rb64 = I.Csr(b.nrows, b.ncols, b.row_ptr, b.col, b.val.astype(dtype).astype(np.float64))
    ref = oracle.spgemm(ra64, rb64)
    ra, rb = oracle.backward(ra64, rb64, ref.row_ptr, ref.col, dc.astype(np.float64))
    mag = [I.Csr(m.nrows, m.ncols, m.row_ptr, m.col, np.abs(m.val)) for m in (ra64, rb64)]
    ba, bb = oracle.backward(*mag, ref.row_ptr, ref.col, np.abs(dc.astype(np.float64)))
    tol = 1e-12 if tag == "f64" else 1e-5      # of the sum of the terms' magnitudes, as for C
    assert np.all(np.abs(da.double().cpu().numpy() - ra) <= tol * ba)
    assert np.all(np.abs(db.double().cpu().numpy() - rb) <= tol * bb)
