"""Rounds that change nothing are recorded without being run (continuous scores): whole
sweeps that stall, against the FP64 oracle round by round, on each column kernel and in the
batched decoder.

Degrees cover the paired kernels (6, 7, 8), the general ones at their edges (5, 9, 16, 17)
and both score kinds' thresholds: the quantised and noiseless decodes of the same instances
must not look ahead, or stop early, wrongly either (their 0/1 tests are compared with the
oracle round by round elsewhere: FP32 residuals can fall on the other side of a threshold)."""
import numpy as np
import pytest

import gm
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(4099, 1100, 160, 5), (5000, 1000, 200, 6), (6007, 1203, 230, 7), (4096, 900, 160, 8), (3001, 700, 90, 9),
          (2500, 800, 60, 16), (2051, 900, 60, 17), (300, 60, 20, 7)]


def _problem(n, m, k, d, sigma_n, seed):
    I = gm.instance(n, m, k, d, sigma_n, seed)
    y = oracle.sketch(I.rows, I.x.astype(np.float64), m) + I.eta.astype(np.float64)
    return I, y.astype(np.float32)


@pytest.mark.parametrize("mode", ["continuous", "quantised", "noiseless"])
@pytest.mark.parametrize("shape", SHAPES)
def test_stalled_sweeps(shape, mode):
    import paper_1704_09012_gb300 as rl0
    n, m, k, d = shape
    sigma = 0.0 if mode == "noiseless" else 0.02
    I, y = _problem(n, m, k, d, sigma, 40 + d)
    par = dict(sigma_n=sigma, quantised=(mode == "quantised"))
    A = rl0.Expander.from_rows(torch.from_numpy(I.rows).cuda(), m)
    yd = torch.from_numpy(y).cuda()
    x, st = rl0.decode(A, yd, k, **par)
    log = rl0.decode_log(A)
    xo, so, lo = oracle.decode(I.rows, y.astype(np.float64), k, **par)
    assert st["rounds"] == len(log) == so["rounds"]
    if mode == "continuous" and st["rounds"] > 12:
        assert st["skipped_rounds"] > 1
    if mode == "quantised":                           # every round's thresholds differ: none is passed over
        assert st["skipped_rounds"] == 1
    if mode == "continuous":
        for a, b in zip(log, lo):
            assert (a["accepted"], a["updated"]) == (b["accepted"], b["updated"])
            if b["accepted"]:
                assert a["support"] == b["support"]
            assert a["l1_hat"] == pytest.approx(b["l1_hat"], rel=1e-5, abs=1e-3)
        xg = x.cpu().numpy().astype(np.float64)
        assert np.array_equal(np.nonzero(xg)[0], np.nonzero(xo)[0])
        assert np.linalg.norm(xg - xo) <= 1e-5 * np.linalg.norm(xo)
    # the L2-gather kernel (no residual codes) and the batched decoder: the same result
    xs, ss = rl0.decode_static(A, yd, k, **par)
    xb, sb = rl0.decode_batched([A], [yd], [k], par)
    assert torch.equal(xs, x) and torch.equal(xb[0], x)
    for s in (ss, sb[0]):
        assert (s["rounds"], s["accepted_rounds"], s["final_l1"]) == (st["rounds"], st["accepted_rounds"], st["final_l1"])


# (n, m, k, d, sigma_n, seed): sweeps with an update after a stretch of rounds that change nothing
LATE = [(20000, 2000, 220, 7, 0.02, 10), (20000, 2200, 200, 8, 0.02, 0), (16000, 2500, 180, 10, 0.02, 10),
        (12000, 2400, 250, 5, 0.03, 3), (12000, 2400, 250, 5, 0.03, 5)]


@pytest.mark.parametrize("adaptive", [False, True])
@pytest.mark.parametrize("case", LATE)
def test_update_after_idle_rounds(case, adaptive):
    import paper_1704_09012_gb300 as rl0
    n, m, k, d, sigma, seed = case
    I, y = _problem(n, m, k, d, sigma, seed)
    par = dict(sigma_n=sigma, adaptive_k=adaptive)
    A = rl0.Expander.from_rows(torch.from_numpy(I.rows).cuda(), m)
    yd = torch.from_numpy(y).cuda()
    x, st = rl0.decode(A, yd, k, **par)
    log = rl0.decode_log(A)
    xo, so, lo = oracle.decode(I.rows, y.astype(np.float64), k, **par)
    assert [(a["updated"], a["accepted"]) for a in log] == [(b["updated"], b["accepted"]) for b in lo]
    assert [a["k_prior"] for a in log] == pytest.approx([b["k_prior"] for b in lo], rel=1e-4)
    if not adaptive:
        events = [i for i, b in enumerate(lo) if b["updated"]]
        assert max(b - a for a, b in zip(events, events[1:])) > 2
        assert st["skipped_rounds"] > 10
        xb, sb = rl0.decode_batched([A], [yd], [k], par)
        xs, ss = rl0.decode_static(A, yd, k, **par)
        assert torch.equal(xb[0], x) and torch.equal(xs, x)
        assert sb[0]["rounds"] == ss["rounds"] == st["rounds"]
    xg = x.cpu().numpy().astype(np.float64)
    assert np.array_equal(np.nonzero(xg)[0], np.nonzero(xo)[0])
    assert np.linalg.norm(xg - xo) <= 1e-5 * np.linalg.norm(xo)
