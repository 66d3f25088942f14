"""The order of the sums in the scorer's gradient and loss does not depend on the device: the
training code is compiled once more for a device that reports half as many SMs, linked with
the other objects as they are, and run in a child process on the same data.  Sets larger than
one pass of the grid, whose CTAs add several blocks: the same bits."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FAKE = """
#include <cuda_runtime.h>
static cudaError_t half_the_sms(int *v, cudaDeviceAttr a, int dev)
{
    const cudaError_t e = cudaDeviceGetAttribute(v, a, dev);
    if (a == cudaDevAttrMultiProcessorCount) *v /= 2;
    return e;
}
#define cudaDeviceGetAttribute half_the_sms
"""

CHILD = """
import hashlib
import sys
import torch
import paper_1704_09012_gb300 as rl0
rl0.LIB_PATH = sys.argv[1]
g = torch.Generator("cuda").manual_seed(1)
F = torch.randn(150001, 16, generator=g, device="cuda")
y = (torch.rand(150001, generator=g, device="cuda") < 0.4).float()
w = rl0.mlp_init(seed=1)
loss, grad = rl0.mlp_grad(w, F, y)
_, last = rl0.mlp_train(w, F, y, epochs=1, batch=40000)
print(loss.hex(), last.hex(), hashlib.sha256(grad.cpu().numpy().tobytes() + w.cpu().numpy().tobytes()).hexdigest())
"""


def test_bits_do_not_depend_on_the_number_of_sms(tmp_path):
    from paper_1704_09012_gb300 import build
    fake, obj, lib = (str(tmp_path / f) for f in ("fake.h", "mlp.o", "librl0.so"))
    with open(fake, "w") as f:
        f.write(FAKE)
    normal = build.build()
    nv = build.nvcc()
    subprocess.run([nv] + build.ARCH + build.FLAGS + ["-include", fake, "-c", os.path.join(build.CSRC, "rl0_mlp.cu"),
                                                      "-o", obj], check=True)
    objs = [os.path.join(build.OUT, s.replace(".cu", ".o")) for s in build.SOURCES if s != "rl0_mlp.cu"]
    subprocess.run([nv] + build.ARCH + ["-shared", "-o", lib] + objs + [obj, "-cudart", "static"], check=True)
    out = [subprocess.run([sys.executable, "-c", CHILD, p], cwd=build.ROOT, capture_output=True, text=True, timeout=120)
           for p in (normal, lib)]
    assert all(o.returncode == 0 for o in out), out[1].stderr
    assert out[0].stdout == out[1].stdout != ""
