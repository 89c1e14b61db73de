"""Compression of rows around the lines between its kernels (128 entries: a
thread or a warp; 256: a warp or a block) and around the warps' steps of 128
entries, sorted and in any order, with runs that cross a step, against a plain
restatement; and columns out of range in either kind of row."""
import numpy as np
import pytest

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu

LENS = [0, 1, 127, 128, 129, 130, 255, 256, 257, 383, 384, 385, 511, 512, 513, 1023, 1024, 1025, 1026, 2047, 2048, 2049, 3000]


def _matrix(order, seed):
    rng = np.random.default_rng(seed)
    ncols = 40_000
    rows = []
    for n in LENS * 3 + [int(x) for x in rng.integers(100, 1200, size=200)]:
        if rng.random() < 0.5:   # dense stretches: runs of many entries
            c0 = rng.integers(0, ncols - 4 * max(n, 1))
            r = np.sort(c0 + rng.choice(2 * max(n, 1), size=n, replace=False))
        else:
            r = np.sort(rng.choice(ncols, size=n, replace=False))
        if order == "any":
            r = rng.permutation(r)
        elif order == "steps":   # sorted but for one swap across the step at 128
            if n > 130:
                r[[127, 128]] = r[[128, 127]]
        rows.append(r)
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    return I.Csr(len(rows), ncols, rp, np.concatenate(rows).astype(np.int32), np.ones(rp[-1]))


@pytest.mark.parametrize("order", ["sorted", "any", "steps"])
def test_rows(cuda_lib, order):
    m = _matrix(order, 3)
    h = sg.Handle()
    cnt, pairs = h.compress(to_dev(m))
    h.check()
    cnt, pairs = cnt.cpu().numpy(), pairs.cpu().numpy().view(np.uint32)
    for k in range(m.nrows):
        c = m.col[m.row_ptr[k]:m.row_ptr[k + 1]].astype(np.int64)
        cut = np.flatnonzero(np.diff(c >> 5, prepend=-1))
        assert cnt[k] == len(cut), (k, len(c))
        if len(c) == 0:
            continue
        got = pairs[m.row_ptr[k]:m.row_ptr[k] + len(cut)]
        assert np.array_equal(got[:, 0], (c >> 5)[cut])
        bits = np.uint32(1) << (c & 31).astype(np.uint32)
        assert np.array_equal(got[:, 1], np.bitwise_or.reduceat(bits, cut))


@pytest.mark.parametrize("n", [128, 129, 140, 256, 257, 1025])
@pytest.mark.parametrize("at", ["first", "last", "middle"])
def test_columns_out_of_range(cuda_lib, n, at):
    m = _matrix("sorted", 4)
    k = int(np.flatnonzero(np.diff(m.row_ptr) >= n)[0])
    q = {"first": 0, "last": n - 1, "middle": n // 2}[at]
    h = sg.Handle()
    for bad in (-1, m.ncols):
        m.col[m.row_ptr[k] + q] = bad
        M = to_dev(m)
        with pytest.raises(sg.SpgemmError, match="out of range"):
            h.symbolic(to_dev(I.random_csr(10, m.nrows, 0.5, 1)), M)


def test_rows_past_the_line_cost_their_entries(cuda_lib):
    """Compression of 300,000 rows of 136 entries against as many entries in rows
    of 600: a block for every row past 128 entries took over three times as long."""
    import torch
    h = sg.Handle()

    def ms(n, per):
        col = torch.randint(0, 3_000_000 // per, (n, per), device="cuda") + torch.arange(per, device="cuda") * (3_000_000 // per)
        B = sg.Csr(n, 3_000_000, torch.arange(n + 1, device="cuda") * per, col.reshape(-1).int(),
                   torch.ones(1, device="cuda").expand(n * per))
        A = to_dev(I.random_csr(50, n, 2 / n, 1))
        h.symbolic(A, B)
        h.set_timing(True)
        h.reset_timings()
        for _ in range(5):
            h.symbolic(A, B)
        t = h.timings()
        h.set_timing(False)
        return t["compress"][2] + t["compress_long"][2]

    short, long = ms(300_000, 136), ms(68_000, 600)
    assert short < 1.8 * long, (short, long)
