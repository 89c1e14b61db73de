"""Row counts around the sizes at which the scan and binning of the symbolic
phase change their tiles (256 rows, 131,072 rows, tiles of 1024 rows): offsets
and bins of a product whose rows hold 0 to 40 entries."""
import numpy as np
import pytest
import torch

import paper_1804_00695_gb300 as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 255, 256, 257, 512, 131071, 131072, 131073, 132096, 132097, 300001])
def test_offsets_and_bins(cuda_lib, n):
    rng = np.random.default_rng(n)
    lens = rng.choice([0, 1, 2, 17, 33, 40], size=n)
    width = rng.choice([3, 5000])
    b_rows = [np.arange(k) * width for k in range(41)]       # row k of B: k entries
    dev = torch.device("cuda")

    def csr(rows, ncols, rp, col):
        return sg.Csr(rows, ncols, torch.from_numpy(rp).to(dev), torch.from_numpy(col.astype(np.int32)).to(dev),
                      torch.ones(len(col), dtype=torch.float64, device=dev))

    a = csr(n, 41, np.arange(n + 1, dtype=np.int64), lens)   # row i of C: lens[i] entries
    b = csr(41, 41 * 5000, np.concatenate([[0], np.cumsum(np.arange(41))]).astype(np.int64), np.concatenate(b_rows))
    h = sg.Handle()
    c = h.spgemm(a, b)
    h.check()
    assert np.array_equal(c.row_ptr.cpu().numpy(), np.concatenate([[0], np.cumsum(lens)]))
    assert sum(h.bin_counts()[1][1:]) == np.count_nonzero(lens)
    assert np.array_equal(c.col.cpu().numpy(), np.concatenate([b_rows[k] for k in lens]))
