"""Rows counted over bitmaps in the symbolic phase, at the edges of their
kernels: 31-33 compressed pairs (32-slot map or bitmap), 4095-4097 pairs and
2047-2049 blocks (a warp or a block), more stored entries than a batch of 32,
256, 512 or 1024, and a B of the widths where the block's threads change and
where the bitmap no longer fits shared memory; a column of A out of range; and
the compression of rows of B around its chunks of 1024 entries."""
import numpy as np
import pytest

import oracle
import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, oracle_product, to_dev

pytestmark = pytest.mark.gpu


def _csr(rows, ncols, rng):
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    col = np.concatenate(rows).astype(np.int32) if len(rows) else np.zeros(0, np.int32)
    return I.Csr(len(rows), ncols, rp, col, rng.standard_normal(len(col)))


def _operands(nwords, seed):
    rng = np.random.default_rng(seed)
    b_rows, a_rows = [], []

    def row_of(pairs_per_entry, span, base=None):
        """A row whose entries meet rows of B of these many pairs (columns in
        distinct blocks) spanning `span` blocks; its first block and its last
        are reached."""
        span = min(span, nwords)
        base = int(rng.integers(0, nwords - span + 1)) if base is None else base
        first = len(b_rows)
        for e, p in enumerate(pairs_per_entry):
            blk = base + rng.choice(span, size=min(p, span), replace=False)
            if e == 0 and len(blk) > 1:
                blk = np.unique(np.concatenate([blk[2:], [base, base + span - 1]]))
            b_rows.append(np.sort(blk) * 32 + rng.integers(0, 32, size=len(blk)))
        a_rows.append(first + np.arange(len(pairs_per_entry)))

    for n in (31, 32, 33):
        row_of([n], 500)
        row_of([1] * n, 4000)
    for n in (4095, 4096, 4097):
        row_of([64] * (n // 64) + [n % 64 + 1], 2048)
    for span in (2047, 2048, 2049):
        row_of([40, 3, 0, 50], span)
    for n in (33, 257, 513, 1025):
        row_of([3] * n, nwords)
        row_of([0] * (n - 40) + [2] * 40, 300)
    row_of([5000, 9000, 1], nwords)
    row_of([40], 4000, base=0)
    a_rows.append(np.zeros(0, dtype=np.int64))
    return _csr(a_rows, len(b_rows), rng), _csr(b_rows, 32 * nwords - 5, rng)


@pytest.mark.parametrize("narrow", [1, 0])
@pytest.mark.parametrize("nwords", [4500, 8192, 8193, 24576, 24577, 53248, 53249])
def test_symbolic_bitmaps(cuda_lib, nwords, narrow):
    h = sg.Handle()
    h.set_option(sg.OPT_NARROW, narrow)
    a, b = _operands(nwords, nwords)
    b.col = np.minimum(b.col, b.ncols - 1)
    c = h.spgemm(to_dev(a), to_dev(b))
    h.check()
    assert_matches(c, oracle_product(a, b), "f64")


@pytest.mark.parametrize("narrow", [1, 0])
def test_symbolic_bad_column(cuda_lib, narrow):
    """A stored column of A past B's rows in a row for each kernel: an error,
    and the handle works afterwards."""
    h = sg.Handle()
    h.set_option(sg.OPT_NARROW, narrow)
    a, b = _operands(4500, 3)
    for i in range(a.nrows - 1):
        bad = I.Csr(a.nrows, a.ncols, a.row_ptr, a.col.copy(), a.val)
        bad.col[a.row_ptr[i]] = b.nrows if i % 2 else -1
        with pytest.raises(sg.SpgemmError) as ei:
            h.symbolic(to_dev(bad), to_dev(b))
        assert ei.value.status == 3
    b.col = np.minimum(b.col, b.ncols - 1)
    c = h.spgemm(to_dev(a), to_dev(b))
    h.check()
    assert_matches(c, oracle_product(a, b), "f64")


@pytest.mark.parametrize("step", [1, 5, 40])
def test_compress_chunks(cuda_lib, step):
    """Rows of B of lengths around the long-row limit and the chunks, columns
    `step` apart from an offset, so that runs of a block cross the chunks."""
    rng = np.random.default_rng(step)
    rows = [off + step * np.arange(n) for n in (127, 128, 129, 1023, 1024, 1025, 1055, 2047, 2048, 2049, 5000)
            for off in (0, 7, 31)]
    m = _csr(rows, 5000 * step + 40, rng)
    h = sg.Handle()
    cnt, pairs = h.compress(to_dev(m))
    h.check()
    rp, blk, mask = oracle.compress_rows(m)
    cnt, pairs = cnt.cpu().numpy(), pairs.cpu().numpy().view(np.uint32)
    assert np.array_equal(cnt, np.diff(rp))
    for k in range(m.nrows):
        got = pairs[m.row_ptr[k]:m.row_ptr[k] + cnt[k]]
        assert np.array_equal(got[:, 0], blk[rp[k]:rp[k + 1]].astype(np.uint32))
        assert np.array_equal(got[:, 1], mask[rp[k]:rp[k + 1]])
