"""rl0_posterior_mc at the largest number of columns the library takes (d = 1: no pairs): the
grid's steps over the columns must not pass 2^31."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_largest_number_of_columns():
    import paper_1704_09012_gb300 as rl0
    n, m = (1 << 31) - 1, 1 << 26
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 220 << 30:
        pytest.skip("needs 220 GB of device memory")
    A = rl0.Expander.random(n, m, 1, seed=1)
    g = torch.Generator("cuda").manual_seed(1)
    y0 = torch.randint(0, 2, (m,), generator=g, device="cuda").float()
    yh = y0 + 0.01 * torch.randn(m, generator=g, device="cuda")
    hz, he = rl0.posterior_mc(A, y0, yh, 1000, 0.01, wz_max=0.5, we_max=0.5)
    near = yh.abs() < 0.5
    assert int(hz[:, 0].sum()) == int(near.sum()) and int(hz[:, 1].sum()) == int((near & (y0 == 0)).sum())
    assert not he.any()
    A.free()
