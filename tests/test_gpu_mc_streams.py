"""rl0_posterior_mc only reads the expander's rows: it may run on another stream than a decode
of the same expander, and beside another Monte-Carlo call with other inputs; every result is
the one of the same call made alone."""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_beside_a_decode_and_another_call_on_one_expander():
    import paper_1704_09012_gb300 as rl0
    n, m, k, d, sigma = 200003, 40001, 4000, 7, 0.01
    A = rl0.Expander.random(n, m, d, seed=2)
    g = torch.Generator("cuda").manual_seed(2)
    x = torch.zeros(n, device="cuda")
    x[torch.randperm(n, generator=g, device="cuda")[:k]] = torch.randn(k, generator=g, device="cuda")
    y0, y = rl0.sketch(A, x), rl0.sketch(A, x, sigma_n=sigma, noise_seed=3)
    z0, z = rl0.sketch(A, -2.0 * x), rl0.sketch(A, -2.0 * x, sigma_n=sigma, noise_seed=4)
    want, _ = rl0.decode(A, y, k, sigma_n=sigma)
    counts = [[h.clone() for h in rl0.posterior_mc(A, a, b, k, sigma)] for a, b in ((y0, y), (z0, z))]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    got, decoded, calls = [], [], 200

    def monte_carlo(a, b, s):
        with torch.cuda.stream(s):
            hz, he = (torch.zeros((64, 3), dtype=torch.int64, device="cuda") for _ in range(2))
            for _ in range(calls):
                rl0.posterior_mc(A, a, b, k, sigma, hz=hz, he=he, stream=s)
        got.append((a, hz, he))

    threads = [threading.Thread(target=monte_carlo, args=(a, b, s)) for (a, b), s in zip(((y0, y), (z0, z)), streams)]
    for t in threads:
        t.start()
    for _ in range(20):
        decoded.append(rl0.decode(A, y, k, sigma_n=sigma)[0])
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert all(torch.equal(v, want) for v in decoded)
    assert len(got) == 2
    for a, hz, he in got:
        wz, we = counts[0] if a is y0 else counts[1]
        assert torch.equal(hz, calls * wz) and torch.equal(he, calls * we)
