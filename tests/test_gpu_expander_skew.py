"""Building an expander from rows that crowd into a few: buckets of the transpose with more
entries than a CTA's shared memory holds, up to all of them in one row's bucket, beside empty
ones.  As for uniform rows, a sketch without noise must equal the oracle's bit for bit."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rows(n, m, d, crowd, first, rng):
    """n columns: d distinct rows, a share `crowd` of the columns only from the first ones."""
    rows = np.sort(np.argsort(rng.random((n, 4 * d)), axis=1)[:, :d], axis=1)
    stride = np.where(rng.random(n) < crowd, first // (4 * d), m // (4 * d))
    return (rows * stride[:, None] + (rng.random(n) * stride).astype(np.int64)[:, None]).astype(np.int32)


@pytest.mark.parametrize("n,m,d,crowd,first", [(60001, 9973, 7, 1.0, 28), (60001, 9973, 7, 0.5, 280),
                                               (200003, 50021, 7, 0.3, 2800), (40009, 3001, 16, 1.0, 64)])
def test_crowded_rows(n, m, d, crowd, first):
    import paper_1704_09012_gb300 as rl0
    rng = np.random.default_rng(n + d)
    rows = _rows(n, m, d, crowd, first, rng)
    buckets = min(n * d // 2048, 1000, m)
    per = -(-m // buckets)
    assert np.bincount((rows // per).ravel()).max() > 1.25 * n * d / buckets + 1024
    A = rl0.Expander.from_rows(torch.from_numpy(rows).cuda(), m)
    assert np.array_equal(A.rows().cpu().numpy(), rows)
    dense = rng.standard_normal(n).astype(np.float32)
    for x in (dense, np.where(rng.random(n) < 0.02, dense, np.float32(0.0))):
        y = oracle.sketch(rows, x.astype(np.float64), m).astype(np.float32)
        assert np.array_equal(rl0.sketch(A, torch.from_numpy(x).cuda()).cpu().numpy(), y)
