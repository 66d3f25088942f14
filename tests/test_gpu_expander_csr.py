"""Building an expander: both layouts of A and the CSR of its transpose, which the sketch reads
row by row in ascending column order.  A sketch without noise is an FP64 sum rounded once, so it
must equal the oracle's bit for bit, for a sparse x and for a dense one: a missing, repeated or
misplaced entry, or another order, shows.

Shapes: one and several groups of columns and slices of rows, sizes that divide nothing, each
kernel width (d <= 8, 16, 32), d = m, and rows too long, or too many rows, for the shared counters."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (5, 3, 3), (127, 40, 7), (129, 40, 8), (1001, 333, 9), (4099, 700, 17), (2000, 64, 32),
          (50021, 9973, 7), (60001, 53249, 6), (40003, 110001, 16), (9001, 460000, 5), (30000, 8, 3), (300, 7, 7)]


@pytest.mark.parametrize("shape", SHAPES)
def test_layouts_and_transpose(shape):
    import paper_1704_09012_gb300 as rl0
    n, m, d = shape
    A = rl0.Expander.random(n, m, d, seed=n + d)
    want = oracle.make_expander(n, m, d, n + d)
    assert np.array_equal(A.rows().cpu().numpy(), want)
    B = rl0.Expander.from_rows(torch.from_numpy(want).cuda(), m)
    rng = np.random.default_rng(n)
    dense = rng.standard_normal(n).astype(np.float32)
    sparse = np.where(rng.random(n) < 0.02, dense, np.float32(0.0))
    for x in (dense, sparse):
        y = oracle.sketch(want, x.astype(np.float64), m).astype(np.float32)
        for E in (A, B):
            assert np.array_equal(rl0.sketch(E, torch.from_numpy(x).cuda()).cpu().numpy(), y)


def test_bad_rows_are_refused():
    import paper_1704_09012_gb300 as rl0
    good = np.sort(np.random.default_rng(0).permuted(np.tile(np.arange(50, dtype=np.int32), (300, 1)), axis=1)[:, :6], axis=1)
    for j, s, v in ((0, 0, -1), (299, 5, 50), (131, 3, None), (200, 2, None)):
        bad = good.copy()
        bad[j, s] = bad[j, s - 1] if v is None else v
        with pytest.raises(rl0.Rl0Error) as e:
            rl0.Expander.from_rows(torch.from_numpy(bad).cuda(), 50)
        assert e.value.code == -6
