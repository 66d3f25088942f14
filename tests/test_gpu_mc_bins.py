"""rl0_posterior_mc keeps several copies of its counters, as many as the number of bins leaves
room for; the degrees cover each kernel width and columns without a pair."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [1, 2, 7, 9, 17, 32])
def test_totals_do_not_depend_on_the_binning(d):
    """Every sample in range is counted once whatever the number of bins (and so the number of
    copies of the counters): the totals over the bins are the same whole numbers, and the row and
    pair counts are NumPy's."""
    import paper_1704_09012_gb300 as rl0
    n, m, k, sigma = 5003, 1201, 90, 0.02
    A = rl0.Expander.random(n, m, d, seed=d)
    rng = np.random.default_rng(d)
    x = np.zeros(n, np.float32)
    x[rng.choice(n, k, replace=False)] = rng.standard_normal(k)
    y0 = rl0.sketch(A, torch.from_numpy(x).cuda())
    yh = rl0.sketch(A, torch.from_numpy(x).cuda(), sigma_n=sigma, noise_seed=1)
    totals = []
    for nbins in (1, 64, 192, 193, 1024):
        hz, he = rl0.posterior_mc(A, y0, yh, k, sigma, nbins=nbins, wz_max=1.0, we_max=1.0)
        totals.append((hz.sum(0).tolist(), he.sum(0).tolist()))
    assert all(t == totals[0] for t in totals)
    a, b = yh.cpu().numpy(), y0.cpu().numpy()
    rows = A.rows().cpu().numpy()
    s, l = np.triu_indices(d, 1)
    near = np.abs(a[rows[:, s]] - a[rows[:, l]]) < 1.0
    same = b[rows[:, s]] == b[rows[:, l]]
    assert totals[0][0][:2] == [int((np.abs(a) < 1.0).sum()), int(((np.abs(a) < 1.0) & (b == 0)).sum())]
    assert totals[0][1][:2] == [int(near.sum()), int((near & same).sum())]
