"""The calls whose time matters to a user of this library, with the inputs they meet.

Every case is one public call (or, for "instance", the few calls of one experiment):
  decode    Robust-l0 (arXiv 1704.09012, Algorithm 2) on one instance, device buffers;
            options: quantised scores, adaptive_k, the learned column scorer
  host      the same from and to pinned host buffers
  parallel  Parallel-l0 (Algorithm 1), noiseless
  batched   many instances in one call
  instance  a new expander, its sketch and the decode: one trial of a phase transition
  posterior the Monte-Carlo experiment that compares the posteriors with counts
  train     the scorer's training (Adam on minibatches)

listed() and draw() give cases, prepare() makes a case's inputs on the GPU, run() is one
call, work() its unavoidable traffic, and exact() the same outputs in 64 bits from plain
torch."""
import math
import random

import numpy as np
import torch

import paper_1704_09012_gb300 as rl0


def _sigma(d, rho, snr_db):
    """Noise std for a per-measurement SNR: E[y_i^2] = d rho for N(0, 1) signals."""
    return math.sqrt(d * rho) * 10.0 ** (-snr_db / 20.0)


def _case(path, n, delta, rho, d=7, snr=40.0, sigma=None, **options):
    m = max(int(delta * n), d + 1)
    k = max(int(rho * m), 1)
    sigma_n = _sigma(d, k / m, snr) if sigma is None else sigma
    return dict(path=path, n=n, m=m, k=k, d=d, sigma_n=sigma_n, **options)


def listed():
    n20, n22, n24 = 1 << 20, 1 << 22, 1 << 24
    return [
        # one small instance: the latency of a call
        dict(name="small", path="decode", n=4096, m=1024, k=100, d=7, sigma_n=1e-3),
        # the adaptive_k variant (the prior follows the support found) at a mid size that divides
        # nothing, and a degree without kernels of its own
        dict(_case("decode", 100003, 0.2, 0.07, d=10, adaptive=True), name="adaptive"),
        # the benchmark's decode
        dict(_case("decode", n20, 0.1, 0.1), name="large"),
        # its quantised variant in a host program: sketch and result in pinned host memory
        dict(_case("host", n20, 0.1, 0.1, quantised=True), name="host"),
        # Algorithm 1 on an exact sketch, odd sizes
        dict(_case("parallel", 700001, 0.15, 0.08, d=8, sigma=0.0), name="parallel"),
        # more rows than one SM's shared memory holds codes for; past the transition, a whole sweep
        dict(_case("decode", n22, 0.1, 0.15, snr=30.0), name="wide"),
        # the learned scorer on that workload
        dict(_case("decode", n22, 0.1, 0.15, snr=30.0, learned=True), name="learned"),
        # the largest size of the extreme-subsampling experiment
        dict(_case("decode", n24, 0.01, 0.1, sigma=0.01), name="extreme"),
        # a trial of that experiment at its smaller size: every trial draws its own expander
        dict(_case("instance", n22, 0.01, 0.1, sigma=0.001), name="trial"),
        # many mixed instances, served in one call
        dict(path="batched", count=256, n_lo=1 << 10, n_hi=1 << 16, d=7, shape_seed=1, name="batched"),
        # the posteriors against counts at the settings of the paper's figure
        dict(_case("posterior", n20, 0.3, 0.1, sigma=0.01), name="posterior"),
        # training the scorer on some of a decode's candidates
        dict(path="train", rows=400003, epochs=2, batch=4096, name="train"),
    ]


def draw(rng):
    path = rng.choice(["decode", "decode", "decode", "decode", "host", "parallel", "batched", "instance", "posterior",
                       "train"])
    size = lambda lo, hi: int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))
    if path == "train":
        return dict(path=path, rows=size(20000, 400000), epochs=rng.randint(1, 2), batch=rng.choice([2048, 4096, 8192]))
    if path == "batched":
        lo = size(1 << 10, 1 << 13)
        return dict(path=path, count=size(16, 256), n_lo=lo, n_hi=8 * lo, d=rng.choice([6, 7, 8, 10]),
                    shape_seed=rng.randrange(1 << 30))
    hi = {"decode": 1 << 22, "host": 1 << 21, "parallel": 1 << 21, "instance": 1 << 21, "posterior": 1 << 20}[path]
    options = {}
    d = rng.choice([5, 6, 7, 7, 7, 8, 9, 12])
    if path == "decode":
        option = rng.choice(["", "", "quantised", "adaptive", "learned"])
        if option:
            options[option] = True
        if option in ("adaptive", "learned"):
            hi = 1 << 20
    if path in ("host", "instance") and rng.random() < 0.5:
        options["quantised"] = True
    delta = rng.uniform(0.05, 0.3) if rng.random() < 0.7 else rng.uniform(0.005, 0.05)
    rho = rng.uniform(0.05, 0.12) * 7 / d           # d rho decides whether columns can be told apart
    if path == "parallel":
        return _case(path, size(1 << 12, hi), delta, rho, d=d, sigma=0.0)
    return _case(path, size(1 << 12, hi), delta, rho, d=d, snr=rng.uniform(30.0, 60.0), **options)


# ---- inputs --------------------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _rows(n, m, d, gen):
    """d distinct uniform rows per column, ascending: int32 [n, d]."""
    rows = torch.randint(0, m, (n, d), generator=gen, device="cuda", dtype=torch.int32).sort(dim=1).values
    while True:
        bad = (rows[:, 1:] == rows[:, :-1]).any(dim=1).nonzero().flatten()
        if not bad.numel():
            return rows.contiguous()
        again = torch.randint(0, m, (bad.numel(), d), generator=gen, device="cuda", dtype=torch.int32)
        rows[bad] = again.sort(dim=1).values


def _signal(n, k, gen):
    x = torch.zeros(n, device="cuda")
    x[torch.randperm(n, generator=gen, device="cuda")[:k]] = torch.randn(k, generator=gen, device="cuda")
    return x


def _sketch(rows, x, m, sigma_n, gen):
    """A x + eta: A x in integers of 2^-40, so that no order of the additions shows."""
    j = x.nonzero().flatten()
    xi = (x[j].double() * 2.0 ** 40).round().long()
    y = torch.zeros(m, dtype=torch.int64, device="cuda")
    y.index_add_(0, rows[j].long().flatten(), xi[:, None].expand(-1, rows.shape[1]).flatten())
    y = y.double() * 2.0 ** -40
    if sigma_n > 0:
        y = y + sigma_n * torch.randn(m, generator=gen, device="cuda", dtype=torch.float64)
    return y.float()


def _instance(c, seed):
    gen = _generator(seed)
    rows = _rows(c["n"], c["m"], c["d"], gen)
    x = _signal(c["n"], c["k"], gen)
    return rows, x, _sketch(rows, x, c["m"], c["sigma_n"], gen)


def _shapes(c):
    """Mixed instances: n over [n_lo, n_hi], delta in [0.1, 0.3], rho in [0.05, 0.2], SNR 30-60 dB."""
    rng = random.Random(c["shape_seed"])
    return [_case("decode", rng.randint(c["n_lo"], c["n_hi"]), rng.uniform(0.1, 0.3), rng.uniform(0.05, 0.2), d=c["d"],
                  snr=rng.uniform(30.0, 60.0)) for _ in range(c["count"])]


def _padded(c):
    return -(-c["n"] // 64) * 64                    # each x_hat of a batch on its own 256 bytes


def _network(d):
    """A scorer of the kind training gives: the consensus score and the l1 gain count for a
    candidate, its third-smallest deviation against it; the other units carry small weights."""
    gen = torch.Generator().manual_seed(7)
    w1 = 0.02 * torch.randn(16, 32, generator=gen)
    w2 = 0.02 * torch.randn(32, 32, generator=gen)
    w3 = 0.02 * torch.randn(32, generator=gen)
    for unit, (feature, weight) in enumerate([(13, 1.0), (10, 1.0), (2, 0.25)]):
        w1[feature, unit] = weight
        w2[unit, unit] = 1.0
    w3[0], w3[1], w3[2] = 24.0, 4.0, -4.0
    zero = torch.zeros(32)
    w = torch.cat([w1.flatten(), zero, w2.flatten(), zero, w3, torch.tensor([-24.0 * 2.8 / d])])
    return w.to(torch.bfloat16).view(torch.int16).cuda()


def _training_rows(c, seed):
    """Candidates as the decodes log them: sorted deviations, scores, gain, t, d rho; three in
    ten are true, and those have more rows near the consensus value."""
    gen = _generator(seed)
    n = c["rows"]
    u = lambda *s: torch.rand(*s, generator=gen, device="cuda")
    label = (u(n) < 0.3).float()
    spread = torch.where(label > 0, 1.0, 4.0)[:, None] * (0.3 + 1.4 * u(n, 7))
    dev = (torch.randn(n, 7, generator=gen, device="cuda").abs() * spread).clamp(max=8.0).sort(dim=1).values
    ne = (1.0 + torch.exp(-0.5 * dev[:, 1:] ** 2).sum(dim=1)) / 7
    nz = u(n) * 0.3
    gain = (0.6 * label + 0.8 * u(n) - 0.3).clamp(-1.0, 1.0)
    cols = [ne, nz, 0.2 * torch.log1p(300.0 * u(n)), gain, u(n), 0.7 + 0.7 * u(n), ne - nz, torch.zeros_like(ne),
            torch.zeros_like(ne)]
    return torch.cat([dev, torch.stack(cols, dim=1)], dim=1).contiguous(), label


def _first_weights(seed):
    """He-normal weights, zero biases, in the library's order: W1, b1, W2, b2, w3, b3."""
    gen = _generator(seed)
    g = lambda n, fan_in: torch.randn(n, generator=gen, device="cuda") * math.sqrt(2.0 / fan_in)
    zero = torch.zeros(32, device="cuda")
    return torch.cat([g(16 * 32, 16), zero, g(32 * 32, 32), zero, g(32, 32), zero[:1]])


# ---- a call --------------------------------------------------------------------------------

def _options(c):
    o = dict(sigma_n=c["sigma_n"])
    if c.get("quantised"):
        o["quantised"] = True
    if c.get("adaptive"):
        o["adaptive_k"] = True
    return o


def prepare(case, seed):
    path = case["path"]
    state = dict(case=case)
    if path == "train":
        state["features"], state["labels"] = _training_rows(case, seed)
        state["start"] = _first_weights(seed)
    elif path == "batched":
        shapes = _shapes(case)
        made = [_instance(s, seed * 4099 + i) for i, s in enumerate(shapes)]
        As = [rl0.Expander.from_rows(rows, s["m"]) for s, (rows, _, _) in zip(shapes, made)]
        state["x"] = torch.zeros(sum(_padded(s) for s in shapes), device="cuda")
        outs = [x[:s["n"]] for s, x in zip(shapes, state["x"].split([_padded(s) for s in shapes]))]
        state["plan"] = rl0.BatchPlan(As, [y for _, _, y in made], [s["k"] for s in shapes],
                                      [_options(s) for s in shapes], outs)
    elif path == "instance":
        state["x"] = _signal(case["n"], case["k"], _generator(seed))
        state["seed"] = seed
    else:
        rows, x, y = _instance(case, seed)
        state["A"] = rl0.Expander.from_rows(rows, case["m"])
        state["y"] = y.cpu().pin_memory() if path == "host" else y
        state["options"] = _options(case)
        if path == "posterior":
            state["y0"] = _sketch(rows, x, case["m"], 0.0, None)
        if case.get("learned"):
            state["options"].update(scorer=1, mlp=_network(case["d"]), mlp_threshold=0.5)
        if path == "host":
            state["out"] = torch.empty(case["n"], pin_memory=True)
    return state


def _decoded(x, stats):
    return dict(x=x, final_l1=stats["final_l1"], rounds=stats["rounds"], accepted=stats["accepted_rounds"],
                support=stats["support_size"], converged=stats["converged"])


def run(state):
    case = state["case"]
    path = case["path"]
    if path == "decode":
        return _decoded(*rl0.decode(state["A"], state["y"], case["k"], **state["options"]))
    if path == "host":
        return _decoded(*rl0.decode_host(state["A"], state["y"], case["k"], out=state["out"], **state["options"]))
    if path == "parallel":
        return _decoded(*rl0.parallel_l0(state["A"], state["y"]))
    if path == "batched":
        _, stats = state["plan"].run()
        return dict(x=state["x"], final_l1=np.array([s["final_l1"] for s in stats]),
                    rounds=np.array([s["rounds"] for s in stats]))
    if path == "instance":
        A = rl0.Expander.random(case["n"], case["m"], case["d"], seed=state["seed"])
        y = rl0.sketch(A, state["x"], sigma_n=case["sigma_n"], noise_seed=state["seed"] + 7)
        out = _decoded(*rl0.decode(A, y, case["k"], **_options(case)))
        A.free()
        return dict(out, y=y)
    if path == "posterior":
        rows, pairs = rl0.posterior_mc(state["A"], state["y0"], state["y"], case["k"], case["sigma_n"])
        return dict(rows=rows, pairs=pairs)
    w = state["start"].clone()
    bf16, loss = rl0.mlp_train(w, state["features"], state["labels"], epochs=case["epochs"], batch=case["batch"])
    return dict(weights=w, bf16=bf16, loss=loss)


def work(case):
    """One reading of A, y and the other inputs and one writing of the outputs; one multiply-add
    per nonzero of A (the rounds a decode takes depend on its data), or the network's arithmetic."""
    path = case["path"]
    if path == "train":
        params = 16 * 32 + 32 * 32 + 32
        rows = case["rows"]
        # three products per weight and row and epoch, and the loss of the final weights
        return dict(bytes=68 * rows * (case["epochs"] + 1) + 10 * 1633,
                    flops=rows * params * (6 * case["epochs"] + 2))
    if path == "batched":
        parts = [work(s) for s in _shapes(case)]
        return dict(bytes=sum(p["bytes"] for p in parts), flops=sum(p["flops"] for p in parts))
    n, m, d = case["n"], case["m"], case["d"]
    if path == "posterior":
        return dict(bytes=4 * n * d + 8 * m + 2 * 64 * 24, flops=n * d * (d - 1) // 2)
    return dict(bytes=4 * n * d + 4 * m + 4 * n + (4 * m if path == "instance" else 0), flops=2 * n * d)


# ---- the same in 64 bits -------------------------------------------------------------------

def _series(lam, vn, ell=4):
    """1 / p = sum of a_q exp(b_q w^2): Poisson weights lam^q / q!, variances q + vn, the tail
    q > ell as one term of matched variance, normalised at w = 0."""
    terms = [lam ** q / math.factorial(q) for q in range(ell + 100)]
    tail, tail1 = sum(terms[ell + 1:]), sum(terms[ell:])
    w, v = terms[:ell + 1] + [tail], [q + vn for q in range(ell + 1)] + [(lam * tail1 + vn * tail) / tail]
    a = [wq * math.sqrt(vn / vq) for wq, vq in zip(w, v)]
    return [(aq / sum(a), 0.5 / vn - 0.5 / vq) for aq, vq in zip(a, v)]


def _inverse_p(series, w):
    u = w * w
    return sum(a * torch.exp(b * u) for a, b in series)


def _columns(x, n):
    """Ranges of columns whose d x d arrays fit comfortably."""
    return [(j, min(n, j + x)) for j in range(0, n, x)]


def _residual(rows, x, y):
    j = x.nonzero().flatten()
    return y.index_add(0, rows[j].long().flatten(), -x[j][:, None].expand(-1, rows.shape[1]).flatten())


def _updates(rows, r, anchor, qz, qe, alpha):
    """Algorithm 2's loop over columns and anchors: the last passing anchor's consensus value."""
    n, d = rows.shape
    u = torch.zeros(n, dtype=torch.float64, device=r.device)
    for lo, hi in _columns(1 << 20, n):
        idx = rows[lo:hi].long()
        nz = qz[idx].sum(dim=1)
        j = (anchor[idx].any(dim=1) & (d - nz >= alpha)).nonzero().flatten()   # n_e is at most d
        idx, nz = idx[j], nz[j]
        R = r[idx]
        q = qe(R[:, :, None] - R[:, None, :])
        ne = q.sum(dim=2)
        w = (R[:, None, :] * q).sum(dim=2) / ne
        lhs = (R[:, None, :] - w[:, :, None]).abs().sum(dim=2)
        ok = anchor[idx] & (lhs <= R.abs().sum(dim=1)[:, None]) & (ne - nz[:, None] >= alpha)
        last = (ok * torch.arange(1, d + 1, device=r.device)).max(dim=1).values
        u[lo + j] = torch.where(last > 0, w.gather(1, (last - 1).clamp(min=0)[:, None])[:, 0], 0.0)
    return u


def _keep_largest(x, k):
    j = x.nonzero().flatten()
    if j.numel() <= k:
        return x
    order = torch.sort(x[j].abs(), descending=True, stable=True).indices
    x = x.clone()
    x[j[order[k:]]] = 0.0
    return x


def _algorithm2(c, rows, y):
    n, m, k, d, sn = c["n"], c["m"], c["k"], c["d"], c["sigma_n"]
    delta, rho, quantised = m / n, k / m, bool(c.get("quantised"))
    if delta <= 0.05:
        step = 0.01
    else:
        step = (0.05 if rho <= 0.1 else 0.075 if rho <= 0.2 else 0.1) if quantised else 0.025
    alpha = d // 2 + 1 if quantised else 0.5 * d
    y = y.double()
    x, r, l1 = torch.zeros(n, dtype=torch.float64, device=y.device), y, y.abs().sum().item()
    stop, prior = m * sn * math.sqrt(2.0 / math.pi), float(k)
    for index in range(1, math.ceil(1.0 / step - 1e-9)):     # t = 1 changes nothing when there is noise
        if l1 <= stop:
            break
        t = 1.0 - index * step
        pz, pe = _series(d * prior / m, sn * sn), _series(2 * d * prior / m, 2 * sn * sn)
        fz = _inverse_p(pz, r)
        if quantised:
            qz, qe = (fz <= 1.0 / (1.0 - t)).double(), lambda D: (_inverse_p(pe, D) <= 1.0 / t).double()
        else:
            qz, qe = 1.0 / fz, lambda D: 1.0 / _inverse_p(pe, D)
        new = _keep_largest(x + _updates(rows, r, fz >= 1.0 / (1.0 - t), qz, qe, alpha), k)
        rn = _residual(rows, new, y)
        if rn.abs().sum().item() < l1:
            x, r, l1 = new, rn, rn.abs().sum().item()
            if c.get("adaptive"):
                v = x[x != 0]
                prior = max(k - (1.0 - 1.0 / _inverse_p(pz, v)).sum().item(), math.floor(m / 100))
    return x, l1


def _algorithm1(c, rows, y, tol=1e-5):
    y = y.double()
    x, r = torch.zeros(c["n"], dtype=torch.float64, device=y.device), y
    for _ in range(100):
        zero = r.abs() <= tol
        u = _updates(rows, r, ~zero, zero.double(), lambda D: (D.abs() <= tol).double(), c["d"] // 2 + 1)
        if not u.any():
            break
        x = x + u
        r = _residual(rows, x, y)
    return x


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10: four 32-bit words per counter, in int64 tensors."""
    low, k0, k1 = 0xFFFFFFFF, seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (p1 >> 32 & low) ^ c1 ^ k0, p1 & low, (p0 >> 32 & low) ^ c3 ^ k1, p0 & low
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    return c0, c1, c2, c3


def _drawn_rows(n, m, d, seed):
    """Expander.random's matrix: words to [0, m) by multiply-shift with rejection, repeats skipped."""
    j = torch.arange(n, device="cuda")
    rows = torch.full((n, d), -1, dtype=torch.int64, device="cuda")
    got = torch.zeros_like(j)
    block, zero = 0, torch.zeros_like(j)
    while bool((got < d).any()):
        for word in _philox(zero + block, j, zero, zero + 0x41, seed):
            p = word * m
            value = p >> 32
            take = ((p & 0xFFFFFFFF) >= (2 ** 32 - m) % m) & (got < d) & ~(rows == value[:, None]).any(dim=1)
            i = take.nonzero().flatten()
            rows[i, got[i]] = value[i]
            got += take
        block += 1
    return rows.sort(dim=1).values.int()


def _drawn_sketch(rows, x, m, sigma_n, seed):
    y = -_residual(rows, x.double(), torch.zeros(m, dtype=torch.float64, device="cuda"))
    i = torch.arange(m, device="cuda")
    zero = torch.zeros_like(i)
    a, b, _, _ = _philox(zero, i, zero, zero + 0x4E, seed)
    z = torch.sqrt(-2.0 * torch.log((a.double() + 1.0) / 2.0 ** 32)) * torch.cos(2.0 * math.pi * b.double() / 2.0 ** 32)
    return y + sigma_n * z


def _trained(c, features, labels, w):
    """Adam (b1 0.9, b2 0.999, eps 1e-8, rate 3e-3) on the mean cross-entropy of consecutive rows."""
    F, Y, w = features.double(), labels.double(), w.double()

    def loss(w, F, Y):
        w1, b1, w2, b2, w3, b3 = w.split([512, 32, 1024, 32, 32, 1])
        h = torch.relu(torch.relu(F @ w1.view(16, 32) + b1) @ w2.view(32, 32) + b2)
        return torch.nn.functional.binary_cross_entropy_with_logits(h @ w3 + b3, Y)

    m, v, step = torch.zeros_like(w), torch.zeros_like(w), 0
    for _ in range(c["epochs"]):
        for lo in range(0, len(Y), c["batch"]):
            p = w.clone().requires_grad_()
            g, = torch.autograd.grad(loss(p, F[lo:lo + c["batch"]], Y[lo:lo + c["batch"]]), p)
            step += 1
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            w = w - 3e-3 * (m / (1 - 0.9 ** step)) / ((v / (1 - 0.999 ** step)).sqrt() + 1e-8)
    return w, loss(w, F, Y).item()


def _solved(x, l1):
    return dict(x=x, final_l1=l1, rounds=None, accepted=None, support=None, converged=None)


def exact(case, seed):
    path = case["path"]
    if path == "posterior" or case.get("learned"):
        return None                                 # whole numbers; two sweeps over every candidate: too long
    if path == "train":
        features, labels = _training_rows(case, seed)
        w, loss = _trained(case, features, labels, _first_weights(seed))
        return dict(weights=w, bf16=None, loss=loss)
    if path == "batched":
        xs, l1s = [], []
        for i, s in enumerate(_shapes(case)):
            rows, _, y = _instance(s, seed * 4099 + i)
            x, l1 = _algorithm2(s, rows, y)
            xs.append(torch.nn.functional.pad(x, (0, _padded(s) - s["n"])))
            l1s.append(l1)
        return dict(x=torch.cat(xs), final_l1=np.array(l1s), rounds=None)
    if path == "instance":
        rows = _drawn_rows(case["n"], case["m"], case["d"], seed)
        x = _signal(case["n"], case["k"], _generator(seed))
        y = _drawn_sketch(rows, x, case["m"], case["sigma_n"], seed + 7)
        return dict(_solved(*_algorithm2(case, rows, y.float())), y=y)
    rows, _, y = _instance(case, seed)
    if path == "parallel":
        # the residual left is the rounding of y and x_hat to 32 bits, not a value to compare with
        return _solved(_algorithm1(case, rows, y), None)
    return _solved(*_algorithm2(case, rows, y))
