"""Where the resident-code kernel keeps the learned scorer's network in shared memory: beside the
codes when they leave room for it, in the resolve's scratch when they do not (m between
about 112 400 and 114 100), and with few survivors staged beside it (m just below).  Learned round
steps on either side of each edge, in a paired and a general degree, against the FP64 oracle."""
import numpy as np
import pytest

import gm
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _network(d):
    """The consensus score and the l1 gain count for a candidate, its third-smallest deviation
    against it; the other units carry small weights."""
    rng = np.random.default_rng(7)
    w1, w2, w3 = (0.02 * rng.standard_normal(s).astype(np.float32) for s in ((16, 32), (32, 32), 32))
    for unit, (feature, weight) in enumerate([(13, 1.0), (10, 1.0), (2, 0.25)]):
        w1[feature, unit] = weight
        w2[unit, unit] = 1.0
    w3[:3] = 24.0, 4.0, -4.0
    b1 = 0.05 * rng.standard_normal(32).astype(np.float32)
    b2 = 0.05 * rng.standard_normal(32).astype(np.float32)
    return np.concatenate([w1.ravel(), b1, w2.ravel(), b2, w3, np.float32([-24.0 * 2.8 / d])])


@pytest.mark.parametrize("n,m,d", [(5001, 1203, 7), (300001, 112200, 7), (300001, 112392, 7), (300001, 112393, 8),
                                   (300001, 114128, 7), (120001, 113500, 12), (120001, 30000, 12)])
def test_learned_round_step(n, m, d):
    import paper_1704_09012_gb300 as rl0
    k = max(1, int(0.1 * m))
    sigma = gm.sigma_from_snr(d, k / m, 30.0)
    I = gm.instance(n, m, k, d, sigma, 77 + d)
    y = (oracle.sketch(I.rows, I.x.astype(np.float64), m) + I.eta.astype(np.float64)).astype(np.float32)
    rng = np.random.default_rng(d)
    x = I.x.astype(np.float64).copy()
    x[rng.choice(I.support, k // 2, replace=False)] = 0.0
    sh = rng.choice(I.support, k // 5, replace=False)
    x[sh] += rng.choice([-1, 1], sh.size) * rng.uniform(0.2, 1.0, sh.size)
    x = x.astype(np.float32)
    r = (y.astype(np.float64) - oracle.sketch(I.rows, x.astype(np.float64), m)).astype(np.float32)
    wb = rl0.mlp_export(torch.from_numpy(_network(d)).cuda())
    A = rl0.Expander.from_rows(torch.from_numpy(I.rows).cuda(), m)
    with oracle.openmp():
        xo, ro, _, rec = oracle.round_step(I.rows, y.astype(np.float64), k, 8, x.astype(np.float64), r.astype(np.float64),
                                           sigma_n=sigma, mlp_bf16=wb.cpu().numpy().view(np.uint16))
    xg, rg, passed, l1 = rl0.round_step(A, torch.from_numpy(y).cuda(), k, 8, torch.from_numpy(x).cuda(),
                                        torch.from_numpy(r).cuda(), sigma_n=sigma, scorer=1, mlp=wb)
    pg, po = passed.cpu().numpy().astype(bool), rec["passed"].astype(bool)
    near = rec["min_margin"] < 1e-3
    assert po.sum() > k // 20 and near.sum() <= 3 + n // 1000
    assert np.array_equal(pg[~near], po[~near])
    if np.array_equal(pg, po):
        xg = xg.cpu().numpy().astype(np.float64)
        assert np.array_equal(np.nonzero(xg)[0], np.nonzero(xo)[0])
        assert np.linalg.norm(xg - xo) <= 1e-5 * np.linalg.norm(xo)
        assert l1 == pytest.approx(np.abs(ro).sum(), rel=1e-6)
