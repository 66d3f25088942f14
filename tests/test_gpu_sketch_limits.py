"""The sketch of an expander with almost 2^31 entries, the most the library takes: the last
rows' places in the CSR lie within a row's length of 2^31, so 32-bit arithmetic on them must
not run past it.  x holds small whole numbers: every sum is exact in any order."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_sketch_next_to_the_largest_number_of_entries():
    import paper_1704_09012_gb300 as rl0
    n, m, d = (1 << 26) - 1, 1 << 25, 32                # n d = 2^31 - 32
    if torch.cuda.mem_get_info()[0] < 100 << 30:
        pytest.skip("needs 100 GB of device memory")
    A = rl0.Expander.random(n, m, d, seed=1)
    x = torch.randint(-3, 4, (n,), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    y = rl0.sketch(A, x.float())
    rows = A.rows()
    A.free()
    want = torch.zeros(m, device="cuda", dtype=torch.float64)
    for s in range(d):
        want.index_add_(0, rows[:, s].long(), x.double())
    assert torch.equal(y.double(), want)
    del rows, want
    torch.cuda.empty_cache()
