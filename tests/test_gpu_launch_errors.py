"""A column kernel whose launch shape the device refuses is an error, not a decode that
changes nothing.  The library's L2-gather kernels are compiled once more with an occupancy
query that fails, linked with the other objects as they are, and called in a child process:
a decode that needs them returns RL0_ERR_CUDA (graph, profile graph, adaptive, learned,
round step, static workspace); what does not need them works as before."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FAKE = """
#include <cuda_runtime.h>
template <class... A> static cudaError_t refused_query(A...) { return cudaErrorUnknown; }
#define cudaOccupancyMaxActiveBlocksPerMultiprocessor refused_query
"""

CHILD = """
import sys
import torch
import paper_1704_09012_gb300 as rl0
rl0.LIB_PATH = sys.argv[1]


def code(f, *a, **k):
    try:
        f(*a, **k)
    except rl0.Rl0Error as e:
        return e.code
    return 0


def problem(n, m, k):
    A = rl0.Expander.random(n, m, 7, seed=1)
    x = torch.zeros(n, device="cuda")
    x[: k * (n // k) : n // k] = torch.randn(k, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    return A, rl0.sketch(A, x, sigma_n=0.01), x


mlp = rl0.mlp_export(rl0.mlp_init(seed=1))
A, y, x = problem(200000, 120000, 9000)               # too many rows for resident codes
par = dict(sigma_n=0.01)
refused = [code(rl0.decode, A, y, 9000, **par), code(rl0.decode, A, y, 9000, quantised=True, **par),
           code(rl0.decode, A, y, 9000, profile=True, **par), code(rl0.decode, A, y, 9000, adaptive_k=True, **par),
           code(rl0.decode, A, y, 9000, scorer=1, mlp=mlp, **par), code(rl0.parallel_l0, A, y),
           code(rl0.round_step, A, y, 9000, 10, x, y, **par)]
B, yb, xb = problem(4096, 1024, 100)
refused.append(code(rl0.decode_static, B, yb, 100, **par))
works = code(rl0.decode, B, yb, 100, **par)           # the resident-code kernel
xo, st = rl0.decode(B, yb, 100, **par)
torch.cuda.synchronize()
print("refused", refused, "works", works, st["accepted_rounds"] > 0)
"""


def test_a_refused_launch_shape_is_an_error(tmp_path):
    from paper_1704_09012_gb300 import build
    fake, obj, lib = (str(tmp_path / f) for f in ("fake.h", "l2.o", "librl0.so"))
    with open(fake, "w") as f:
        f.write(FAKE)
    build.build()
    nv = build.nvcc()
    subprocess.run([nv] + build.ARCH + build.FLAGS + ["-include", fake, "-c", os.path.join(build.CSRC, "rl0_column_l2.cu"),
                                                      "-o", obj], check=True)
    objs = [os.path.join(build.OUT, s.replace(".cu", ".o")) for s in build.SOURCES if s != "rl0_column_l2.cu"]
    subprocess.run([nv] + build.ARCH + ["-shared", "-o", lib] + objs + [obj, "-cudart", "static"], check=True)
    out = subprocess.run([sys.executable, "-c", CHILD, lib], cwd=build.ROOT, capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stderr
    assert out.stdout.strip() == "refused %s works 0 True" % ([-2] * 8)
