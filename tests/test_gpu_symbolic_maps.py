"""Symbolic phase of rows with few compressed pairs over wide spans: a map of the
row's blocks in place of a bitmap of its span, by a warp (up to 256 pairs) or by
a block (up to 2048, one for 28 blocks).  Rows around every line of the rule and
of the maps' sizes, spans around 2048, 8192, 12,288 and 24,576 blocks and up to the widest
bitmap, counts and columns against the CPU oracle; and such rows must not cost a
pass over their span each."""
import math

import numpy as np
import pytest

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, oracle_product, to_dev

pytestmark = pytest.mark.gpu

SPANS = [2040, 2047, 2048, 2049, 2500, 8191, 8193, 12287, 12288, 12289, 24575, 24576, 24577, 24600, 53248]
PAIRS = [31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 300, 511, 512, 513, 639, 640, 641, 768, 1023, 1024, 1025,
         2000, 2047, 2048, 2049, 2050, 4095, 4097]


def _csr(rows, ncols, rng):
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    return I.Csr(len(rows), ncols, rp, np.concatenate(rows).astype(np.int32), rng.uniform(0.5, 1.5, rp[-1]))


@pytest.mark.parametrize("span", SPANS)
@pytest.mark.parametrize("repeat", [1, 3])
def test_counts(cuda_lib, span, repeat):
    """Row i of A meets pairs[i] pairs over exactly `span` blocks: runs of rows of
    B of 1 to 40 blocks each, the first and the last block of the span among
    them; with repeat 3 every block is met up to three times."""
    rng = np.random.default_rng(span * 10 + repeat)
    ncols = span * 32
    b_rows = [np.array([0]), np.array([ncols - 1])]
    by_len = {}
    for n in (1, 7, 20, 40):
        by_len[n] = []
        for _ in range(220 if n > 1 else 400):
            blocks = np.sort(rng.choice(span, size=n, replace=False))
            cols = blocks * 32 + rng.integers(0, 32, size=n)
            by_len[n].append(len(b_rows))
            b_rows.append(cols)
    a_rows = []
    for want in PAIRS:
        left, ks = want - 2, [0, 1]
        for n in (40, 20, 7, 1):
            take = min(left // n, len(by_len[n]) // repeat if n > 1 else left)
            ks += list(rng.choice(by_len[n], size=min(take, len(by_len[n])), replace=False))
            left -= n * min(take, len(by_len[n]))
        a_rows.append(np.sort(np.array(ks)))
    a, b = _csr(a_rows * repeat, len(b_rows), rng), _csr(b_rows, ncols, rng)
    h = sg.Handle()
    c = h.spgemm(to_dev(a), to_dev(b))
    h.check()
    assert_matches(c, oracle_product(a, b), "f64")


def test_wide_rows_cost_their_pairs(cuda_lib):
    """200,000 rows of about 40 pairs over 50,000 blocks against the same number
    over 2000: a pass over the span took 12 times the map's time."""
    import torch
    rng = np.random.default_rng(5)
    h = sg.Handle()

    def best(blocks):
        n, per = 20000, 20
        b = _csr([np.sort(rng.choice(blocks * 32, size=per, replace=False)) for _ in range(n)], blocks * 32, rng)
        ks = torch.sort(torch.randint(0, n // 2, (200000, 2), device="cuda") + torch.tensor([0, n // 2], device="cuda"))[0]
        rp = torch.arange(0, 400001, 2, device="cuda")
        A = sg.Csr(200000, n, rp, ks.reshape(-1).int(), torch.ones(400000, dtype=torch.float64, device="cuda"))
        B = to_dev(b)
        t = math.inf
        for _ in range(5):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            h.symbolic(A, B)
            e1.record()
            torch.cuda.synchronize()
            t = min(t, e0.elapsed_time(e1))
        return t

    narrow, wide = best(2000), best(50000)
    assert wide < 4 * narrow, (narrow, wide)
