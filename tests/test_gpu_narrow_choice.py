"""How many lanes the narrow rows take: by their own products, whatever the other
rows have, and no more than the rows of B and a wave of the chip can use.  The time
of the narrow kernel against the same rows alone, and against the lanes set by
hand; the products against the oracle."""
import numpy as np
import pytest
import torch

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, host_csr, oracle_product

pytestmark = pytest.mark.gpu


def _csr(parts, ncols, dtype):
    """Rows of equal length each part: (rows, entries, first column, width)."""
    rows, cols, at = [], [], 0
    gen = torch.Generator(device="cuda").manual_seed(len(parts))
    for n, per, lo, width in parts:
        c = torch.randint(0, width // per, (n, per), device="cuda", generator=gen) + torch.arange(per, device="cuda") * (width // per)
        cols.append((c + lo).reshape(-1))
        rows.append(torch.full((n,), per, device="cuda"))
    rp = torch.zeros(sum(len(r) for r in rows) + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.cat(rows), 0, out=rp[1:])
    col = torch.cat(cols).int()
    return sg.Csr(len(rp) - 1, ncols, rp, col, torch.rand(len(col), dtype=dtype, device="cuda", generator=gen) - 0.5)


def _ms(h, a, b):
    rp, nnz = h.symbolic(a, b)
    c = h.numeric(a, b, rp, nnz)
    h.check()
    h.set_timing(True)
    best = 1e9
    for _ in range(5):
        h.reset_timings()
        h.numeric_into(a, b, c)
        best = min(best, h.timings()["numeric.narrow"][2])
    h.set_timing(False)
    return best, c


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_own_products_decide(cuda_lib, dtype):
    """200 rows of 4000 products, alone and among 200,000 wide rows of 8."""
    h = sg.Handle()
    b = _csr([(4000, 8, 0, 32), (20000, 8, 0, 200_000)], 200_000, dtype)
    few = (200, 500, 0, 4000)
    alone, _ = _ms(h, _csr([few], 24000, dtype), b)
    mixed, _ = _ms(h, _csr([few, (200_000, 1, 4000, 20000)], 24000, dtype), b)
    assert mixed < 3 * alone, (alone, mixed)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("rows", [5000, 9000, 12000, 16000, 27000, 38000])
@pytest.mark.parametrize("blen", [3, 8, 24])
def test_no_lanes_by_hand_are_much_better(cuda_lib, dtype, rows, blen):
    h = sg.Handle()
    a, b = _csr([(rows, 2400 // blen, 0, 4000)], 4000, dtype), _csr([(4000, blen, 0, 32)], 32, dtype)
    auto, c = _ms(h, a, b)
    by_hand = []
    for lanes in (4, 8, 16):
        h.set_option(sg.OPT_LANES_NARROW_NUMERIC, lanes)
        t, d = _ms(h, a, b)
        by_hand.append(t)
        assert torch.equal(c.col, d.col) and torch.allclose(c.val, d.val, rtol=0, atol=1e-4 if dtype == torch.float32 else 1e-12)
    assert auto < 1.35 * min(by_hand), (auto, by_hand)


@pytest.mark.parametrize("dtype,tag", [(np.float64, "f64"), (np.float32, "f32")])
@pytest.mark.parametrize("rows", [5300, 5400, 8700, 8800, 10600, 10800, 11000])
@pytest.mark.parametrize("blen", [3, 8, 12])
def test_around_the_lines(cuda_lib, dtype, tag, rows, blen):
    t = torch.float64 if dtype == np.float64 else torch.float32
    a, b = _csr([(rows, 7, 0, 500), (3, 1, 0, 500)], 500, t), _csr([(500, blen, 5, 24)], 40, t)
    c = sg.Handle().spgemm(a, b)
    assert_matches(c, oracle_product(host_csr(a), host_csr(b), dtype), tag)


@pytest.mark.parametrize("rows,alen", [(5000, 60), (9000, 60), (9000, 200), (16000, 30), (25000, 12), (38000, 12)])
def test_symbolic_lanes(cuda_lib, rows, alen):
    """No number of lanes set by hand counts the rows much faster."""
    h = sg.Handle()
    a, b = _csr([(rows, alen, 0, 400)], 400, torch.float32), _csr([(400, 24, 0, 2000)], 2000, torch.float32)

    def ms():
        rp = h.symbolic(a, b)[0]
        h.set_timing(True)
        best = 1e9
        for _ in range(5):
            h.reset_timings()
            h.symbolic(a, b)
            best = min(best, h.timings()["symbolic.narrow"][2])
        h.set_timing(False)
        return best, rp

    auto, rp = ms()
    by_hand = []
    for lanes in (4, 8, 16, 32):
        h.set_option(sg.OPT_LANES_NARROW_SYMBOLIC, lanes)
        t, rp2 = ms()
        by_hand.append(t)
        assert torch.equal(rp, rp2)
    assert auto < 1.3 * min(by_hand), (auto, by_hand)
