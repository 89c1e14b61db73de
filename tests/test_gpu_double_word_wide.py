"""Double-word accumulation of rows over more than 2048 blocks of 32 columns:
outputs around the sizes of the maps (128, 256, 512 and 1024), in lists of the
short rows (products up to 512), the middle ones (1024) and the longer ones,
against the CPU oracle; and rows of at most 128 outputs take the small maps."""
import numpy as np
import pytest

import paper_1804_00695_gb300 as sg
from paper_1804_00695_gb300 import inputs as I
from gpu_helpers import assert_matches, oracle_product, to_dev

pytestmark = pytest.mark.gpu


def _product(outputs, repeat, ncols, rng):
    """Rows of C with exactly these outputs, every product met `repeat` times;
    rows of B of 1 to 9 entries spread over all columns."""
    a_rows, b_rows = [], []
    for n in outputs:
        cols = np.sort(rng.choice(ncols, size=n, replace=False))
        cols[0], cols[-1] = 0, ncols - 1
        cuts = np.unique(np.concatenate([[0, n], np.cumsum(rng.integers(1, 9, size=n))]))
        parts = np.split(cols, cuts[(cuts > 0) & (cuts < n)])
        ks = []
        for _ in range(repeat):
            ks += range(len(b_rows), len(b_rows) + len(parts))
            b_rows += parts
        a_rows.append(np.array(ks))

    def csr(r, m):
        rp = np.concatenate([[0], np.cumsum([len(x) for x in r])]).astype(np.int64)
        return I.Csr(len(r), m, rp, np.concatenate(r).astype(np.int32), rng.standard_normal(rp[-1]))

    return csr(a_rows, len(b_rows)), csr(b_rows, ncols)


@pytest.mark.parametrize("ncols", [70_000, 262_144, 300_000])
@pytest.mark.parametrize("repeat,outputs", [
    (1, [33, 127, 128, 129, 255, 256, 257, 511, 512]), (1, [513, 700, 1000, 1023, 1024]),
    (4, [33, 100, 127, 128]), (2, [128, 129, 255, 256]), (3, [300, 512, 513, 1024]), (5, [128, 256, 512, 900])])
def test_outputs(cuda_lib, ncols, repeat, outputs):
    a, b = _product(outputs * 5, repeat, ncols, np.random.default_rng(repeat * ncols))
    h = sg.Handle()
    h.set_option(sg.OPT_F64_NATIVE, 0)
    h.set_timing(True)
    c = h.spgemm(to_dev(a), to_dev(b))
    h.check()
    assert_matches(c, oracle_product(a, b), "f64")
    t = [k for k in h.timings() if k.startswith("numeric.wide")]
    assert ("numeric.wide4a" in t) == (any(128 < n <= 256 for n in outputs) or (ncols < 300_000 and max(outputs) > 128)), t
    if max(outputs) <= 128:
        assert t == ["numeric.wide3"]
