"""GPU tests of plans on a device part that cannot hold the register tiles at once.

A copy of the library is linked whose cooperative launches all fail with
cudaErrorCooperativeLaunchTooLarge, as on a partition with fewer SMs than the
device reports: every call that would use one still gives its result, on the
first call.
"""
import glob
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FAKE = """
int __wrap_cudaLaunchCooperativeKernel(const void* fn, ...) { return 720; /* cudaErrorCooperativeLaunchTooLarge */ }
"""

CHECK = """
import sys
import torch
from paper_2605_07954_gb300 import _capi
_capi.load(sys.argv[1])
from paper_2605_07954_gb300 import Plan, StencilFn, adjoint, inputs
W = inputs.pattern_weights("heat5")
for shape in ((300, 420), (1000, 1022)):
    x = torch.from_numpy(inputs.field(*shape)).cuda()
    q = Plan(*shape, W, kernel="stream")
    want = q.run(x, 30).double()
    # the kernel that the tiles stand in for, with its bits
    ref = Plan(*shape, W, kernel="resident" if shape[0] == 300 else "stream")
    assert torch.equal(Plan(*shape, W).run(x, 30), ref.run(x, 30))
    for autotune in (False, True, True):
        p = Plan(*shape, W, autotune=autotune)
        for _ in range(2):
            y = p.run(x, 30)
            assert float((y.double() - want).norm() / want.norm()) <= 1e-6, (shape, autotune)
        p.status()
    p = Plan(*shape, W)
    for a, b in zip(adjoint(p, x, x, 12), adjoint(q, x, x, 12)):
        assert float((a.double() - b.double()).norm() / b.double().norm()) <= 1e-6
    p = Plan(*shape, W)
    y, res = p.run_residual(x, 12, 4)
    z, ref = q.run_residual(x, 12, 4)
    assert float((y - z).norm() / z.norm()) <= 1e-6 and torch.allclose(res, ref, rtol=1e-4)
torch.cuda.synchronize()
print("checked")
"""


def test_every_call_works_without_cooperative_launches(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07954_gb300 import build
    build.build()
    objs = sorted(glob.glob(os.path.join(build.BUILD, "*.o")))
    fake, lib = tmp_path / "fake.c", tmp_path / "libfake.so"
    fake.write_text(FAKE)
    subprocess.run([build._nvcc()] + build.ARCH + ["-shared", "-Xcompiler", "-fPIC", "-o", str(lib), str(fake)] + objs
                   + ["-Xlinker", "--wrap=cudaLaunchCooperativeKernel"], check=True)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHECK, str(lib)], cwd=root, env=dict(os.environ, PYTHONPATH=root),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "checked" in r.stdout, r.stdout + r.stderr
