"""The L2-gather column kernel over several chunks per CTA (d = 6, 7, 8; more rows than the
resident-code kernel takes; more than 768 columns per CTA, in numbers that no tile divides):
its ring of survivors carries entries from chunk to chunk, and wraps when many survive.

Round steps from injected residuals, few and many columns passing, in each score kind, against
the FP64 oracle; and whole stalled sweeps, with their passed-over rounds, bit for bit against
the same rounds taken one at a time with rl0_round_step."""
import math

import numpy as np
import pytest

import gm
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N, M, K = 1_500_001, 120_000, 12_000
SIGMA = 0.02
CTAS = 4 * 152                      # at most this many share the columns


@pytest.fixture(scope="module")
def rl0():
    import paper_1704_09012_gb300 as m
    m._lib()
    assert 2 * M > 227 * 1024       # the codes cannot be resident
    return m


_ROWS = {}


def _rows(d):
    if d not in _ROWS:
        _ROWS.clear()
        _ROWS[d] = gm.draw_rows(N, M, d, 60 + d)
    return _ROWS[d]


def _residual(share, sigma, rng):
    """A share of the rows near one value, the others spread over many: a column passes when
    enough of its rows are among the first.  Noiseless: exact multiples of 1/64."""
    r = np.where(rng.random(M) < share, 0.75, rng.integers(-160, 161, M) / 64.0)
    return (r + 0.5 * sigma * rng.standard_normal(M)).astype(np.float32)


@pytest.mark.parametrize("mode", ["continuous", "quantised", "noiseless"])
@pytest.mark.parametrize("d", [6, 7, 8])
def test_round_steps_over_several_chunks(rl0, d, mode):
    rows = _rows(d)
    sigma = 0.0 if mode == "noiseless" else SIGMA
    # a threshold no whole count meets exactly (the quantised default is a count of its own kind)
    par = dict(sigma_n=sigma, quantised=mode == "quantised", alpha=d // 2 + 0.5)
    A = rl0.Expander.from_rows(torch.from_numpy(rows).cuda(), M)
    rng = np.random.default_rng(d)
    x = np.zeros(N, np.float32)
    x[rng.choice(N, 2000, replace=False)] = rng.uniform(0.3, 1.0, 2000)
    y = (oracle.sketch(rows, x.astype(np.float64), M) + rng.standard_normal(M)).astype(np.float32)
    for share, lo, hi in ((0.15, 50, 0.1 * N), (0.62, 4 * 256 * CTAS, N)):
        r = _residual(share, sigma, rng)
        with oracle.openmp():
            _, _, _, rec = oracle.round_step(rows, y.astype(np.float64), K, 10, x.astype(np.float64),
                                             r.astype(np.float64), **par)
        xg, rg, passed, l1 = rl0.round_step(A, torch.from_numpy(y).cuda(), K, 10, torch.from_numpy(x).cuda(),
                                            torch.from_numpy(r).cuda(), **par)
        xg, rg = xg.cpu().numpy().astype(np.float64), rg.cpu().numpy().astype(np.float64)
        pg, po = passed.cpu().numpy().astype(bool), rec["passed"].astype(bool)
        assert lo < po.sum() < hi
        near = rec["min_margin"] < 1e-4
        assert near.sum() < 0.02 * N
        assert np.array_equal(pg[~near], po[~near])
        # x' = H_k(x + updates): the entries kept carry the oracle's values, there are k of
        # them (or all), and none that was dropped is larger (equal ones may change places)
        pre = np.where(pg, x + rec["omega"], x)
        known = ~(near & pg)
        kept = xg != 0.0
        assert abs(int(kept.sum()) - min(K, np.count_nonzero(pre))) <= (pg != po).sum()
        both = kept & known
        assert np.allclose(xg[both], pre[both], rtol=1e-5, atol=4e-6)
        out = known & ~kept & (pre != 0.0)
        if out.any():
            assert np.abs(xg[kept]).min() >= np.abs(pre[out]).max() * (1 - 1e-5) - 4e-6
        # r = y - A x' of that x', rounded as an FP32 sum of a few terms
        want = y.astype(np.float64) - oracle.sketch(rows, xg, M)
        scale = np.abs(y) + oracle.sketch(rows, np.abs(xg), M)
        assert np.all(np.abs(rg - want) <= 16 * scale * 2.0 ** -24 + 1e-30)
        assert l1 == pytest.approx(np.abs(want).sum(), rel=1e-6)


@pytest.mark.parametrize("d", [6, 7, 8])
def test_stalled_sweep_over_several_chunks(rl0, d):
    n, m = 1_200_007, 118_003
    k = int(0.15 * m * 7 / d)
    sigma = gm.sigma_from_snr(d, k / m, 30.0)
    A = rl0.Expander.random(n, m, d, seed=d)
    xt, _ = gm.draw_signal(n, k, 1.0, d)
    y = rl0.sketch(A, torch.from_numpy(xt).cuda(), sigma_n=sigma, noise_seed=d)
    got, st = rl0.decode(A, y, k, sigma_n=sigma)
    log = rl0.decode_log(A)
    assert st["skipped_rounds"] > 3 and st["rounds"] == len(log)
    x, r = torch.zeros(n, device="cuda"), y
    l1 = float(y.double().abs().sum())
    stop = m * sigma * math.sqrt(2.0 / math.pi)
    for i, rec in enumerate(log):
        assert l1 > stop
        xp, rp, passed, l1n = rl0.round_step(A, y, k, i, x, r, sigma_n=sigma)
        updated = int(passed.sum())
        accepted = updated > 0 and l1n < l1
        if accepted:
            x, r, l1 = xp, rp, l1n
        assert (rec["updated"], bool(rec["accepted"])) == (updated, accepted)
        assert rec["l1_hat"] == pytest.approx(l1, rel=1e-12)
    assert l1 <= stop or len(log) == oracle.num_rounds(oracle.default_c(False, m / n, k / m))
    assert torch.equal(x, got)
