"""Workloads for a profiler: each runs one kind of launch of the library inside an NVTX
range of its own name, so that a tool such as Nsight Compute can select it
(--nvtx --nvtx-include "<name>/").

  python -m paper_1704_09012_gb300.profile_workloads round [reps]
      one round of Algorithm 2 at n = 2^20, m = 104857, k = 10485, d = 7, SNR 40 dB
      (the benchmark's instance, expander seed 1000), from the state a decode reaches
      after three rounds, through rl0_round_step, whose column-score and rebuild
      kernels launch directly (outside the decode's conditional graph); `reps`
      repetitions (default 3), each in a range "round";
  python -m paper_1704_09012_gb300.profile_workloads batched [count]
      one rl0_decode_batched call on `count` instances of the batched workload
      (default 256; n uniform in [2^10, 2^16], delta in [0.1, 0.3], rho in [0.05, 0.2],
      d = 7, SNR 30-60 dB), after an untimed call that tunes the schedule, in a range
      "batched";
  python -m paper_1704_09012_gb300.profile_workloads learned [log2n] [reps]
      one learned-scorer round at n = 2^log2n (default 20; 22 is the learned workload's
      evaluation size), m = n/10, rho = 0.15, d = 7, SNR 30 dB, from the state the
      analytic decode reaches after three rounds, through rl0_round_step with a scorer
      trained first on the decode logs of two analytic decodes at n = 2^16 (rl0_scorer_log,
      rl0_mlp_train); `reps` repetitions (default 2), each in a range "learned".  At
      n = 2^20 the round runs on the resident-code kernel, at n = 2^22 (whose codes do not
      fit in shared memory) on the L2-gather kernel.
  python -m paper_1704_09012_gb300.profile_workloads gather [log2n] [reps]
      one round with the analytic rule on the L2-gather kernel: the learned workload's
      instance and state (default n = 2^22), in a range "gather";
  python -m paper_1704_09012_gb300.profile_workloads posterior
      one rl0_posterior_mc call at n = 2^20, m = 0.3 n, rho = 0.1, d = 7, sigma_n = 0.01,
      64 bins, in a range "posterior";
  python -m paper_1704_09012_gb300.profile_workloads train
      rl0_mlp_train on 16384 rows, one pass of 4096-row minibatches, in a range "train";
  python -m paper_1704_09012_gb300.profile_workloads build
      rl0_make_expander at n = 2^22, m = 41943, d = 7, in a range "build".

Every step of the decode runs in the CUDA library; torch only holds device memory and
subtracts A x_hat from y_hat to form the injected residual."""
import sys

import torch

import gm
import paper_1704_09012_gb300 as rl0


def round_workload(reps=3):
    cfg = gm.config_large()
    n, m, k, d, sn = cfg["n"], cfg["m"], cfg["k"], cfg["d"], cfg["sigma_n"]
    A = rl0.Expander.random(n, m, d, seed=1000)
    x, _ = gm.draw_signal(n, k, 1.0, 1000)
    y = rl0.sketch(A, torch.from_numpy(x).cuda(), sigma_n=sn, noise_seed=1001)
    xh, _ = rl0.decode(A, y, k, sigma_n=sn, max_rounds=3)
    rh = y - rl0.sketch(A, xh, sigma_n=0.0)          # r_hat = y_hat - A x_hat
    for _ in range(reps):
        torch.cuda.nvtx.range_push("round")
        rl0.round_step(A, y, k, 3, xh, rh, want_passed=False, sigma_n=sn)
        torch.cuda.nvtx.range_pop()
    torch.cuda.synchronize()


def learned_workload(log2n=20, reps=2):
    from . import learned
    d = 7
    F, Y = [], []
    for i in range(2):
        n = 1 << 16
        m = n // 10
        k = int(0.15 * m)
        sn = gm.sigma_from_snr(d, k / m, 30.0)
        A = rl0.Expander.random(n, m, d, seed=60000 + i)
        x, _ = gm.draw_signal(n, k, 1.0, 60000 + i)
        xt = torch.from_numpy(x).cuda()
        y = rl0.sketch(A, xt, sigma_n=sn, noise_seed=61000 + i)
        f, lab = learned.decode_log_samples(A, y, k, xt, sn)
        F.append(f)
        Y.append(lab)
        A.free()
    wb, _, _ = learned.train_scorer(torch.cat(F), torch.cat(Y), epochs=4)
    _low_snr_round("learned", log2n, reps, scorer=1, mlp=wb)


def gather_workload(log2n=22, reps=2):
    _low_snr_round("gather", log2n, reps)


def _low_snr_round(name, log2n, reps, **params):
    d = 7
    n = 1 << log2n
    m = n // 10
    k = int(0.15 * m)
    sn = gm.sigma_from_snr(d, k / m, 30.0)
    A = rl0.Expander.random(n, m, d, seed=62000)
    x, _ = gm.draw_signal(n, k, 1.0, 62000)
    y = rl0.sketch(A, torch.from_numpy(x).cuda(), sigma_n=sn, noise_seed=63000)
    xh, _ = rl0.decode(A, y, k, sigma_n=sn, max_rounds=3)
    rh = y - rl0.sketch(A, xh, sigma_n=0.0)
    for _ in range(reps):
        torch.cuda.nvtx.range_push(name)
        rl0.round_step(A, y, k, 3, xh, rh, want_passed=False, sigma_n=sn, **params)
        torch.cuda.nvtx.range_pop()
    torch.cuda.synchronize()


def posterior_workload():
    n, d, sn = 1 << 20, 7, 0.01
    m = int(0.3 * n)
    k = int(0.1 * m)
    A = rl0.Expander.random(n, m, d, seed=300)
    x, _ = gm.draw_signal(n, k, 1.0, 300)
    xt = torch.from_numpy(x).cuda()
    y0, y = rl0.sketch(A, xt), rl0.sketch(A, xt, sigma_n=sn, noise_seed=400)
    torch.cuda.nvtx.range_push("posterior")
    rl0.posterior_mc(A, y0, y, k, sn)
    torch.cuda.nvtx.range_pop()
    torch.cuda.synchronize()


def train_workload():
    g = torch.Generator("cuda").manual_seed(1)
    F = torch.randn(16384, 16, generator=g, device="cuda")
    y = (torch.rand(16384, generator=g, device="cuda") < 0.3).float()
    w = rl0.mlp_init(seed=1)
    torch.cuda.nvtx.range_push("train")
    rl0.mlp_train(w, F, y, epochs=1, batch=4096)
    torch.cuda.nvtx.range_pop()


def build_workload():
    torch.cuda.nvtx.range_push("build")
    rl0.Expander.random(1 << 22, 41943, 7, seed=1)
    torch.cuda.nvtx.range_pop()


def batched_workload(count=256):
    shapes = gm.batch_shapes(count, seed=0)
    As, ys, ks, ps = [], [], [], []
    for i, sh in enumerate(shapes):
        A = rl0.Expander.random(sh["n"], sh["m"], sh["d"], seed=50000 + i)
        x, _ = gm.draw_signal(sh["n"], sh["k"], 1.0, 50000 + i)
        ys.append(rl0.sketch(A, torch.from_numpy(x).cuda(), sigma_n=sh["sigma_n"], noise_seed=90000 + i))
        As.append(A)
        ks.append(sh["k"])
        ps.append(dict(sigma_n=sh["sigma_n"]))
    plan = rl0.BatchPlan(As, ys, ks, ps)
    plan.run()
    torch.cuda.synchronize()
    torch.cuda.nvtx.range_push("batched")
    plan.run()
    torch.cuda.nvtx.range_pop()
    torch.cuda.synchronize()


WORKLOADS = {"round": round_workload, "batched": batched_workload, "learned": learned_workload, "gather": gather_workload,
             "posterior": posterior_workload, "train": train_workload, "build": build_workload}


def main(argv):
    if not argv or argv[0] not in WORKLOADS:
        print(__doc__)
        return 2
    torch.cuda.set_device(0)
    WORKLOADS[argv[0]](*[int(v) for v in argv[1:]])
    print("%s workload done" % argv[0])
    return 0


if __name__ == "__main__":
    sys.exit(main(sys.argv[1:]))
