"""GPU tests of the tcgen05 7x7 kernel with four output rows per MMA row: exact
on dyadic data at the edges of its 512-row tiles, against the one-row kernel on
random data, and its bounded waits."""
import numpy as np
import pytest

from paper_2605_07954_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07954_gb300 import build
    build.build()


TYPES = {"bf16": ("tc_bf16", torch.bfloat16, 64), "f32": ("tc_tf32", torch.float32, 96)}


def _plan(shape, W, dtype, phase=True, **kw):
    from paper_2605_07954_gb300 import Plan
    p = Plan(shape[0], shape[1], W, dtype=dtype, compute=TYPES[dtype][0], **kw)
    assert (p.info()["tile_rows"] == 512) == phase, p.info()
    return p


# whole tiles, a last tile of 4 rows / 8 columns, one tile row, many tiles per CTA
SHAPES = [(4096, 4096), (4100, 4104), (8188, 2056), (512, 40000), (2052, 16392)]


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("shape", SHAPES)
def test_dyadic_exact(oracle, dtype, shape):
    """Weights in {0, 1/8} and a 0/1 field, two steps: every product and sum is exact."""
    rng = np.random.default_rng(shape[0] + shape[1])
    W = np.where(rng.random((7, 7)) < 0.7, 0.125, 0.0).astype(np.float32)
    u0 = (rng.random(shape) < 0.5).astype(np.float32)
    x = torch.from_numpy(u0).cuda().to(TYPES[dtype][1])
    p = _plan(shape, W, dtype)
    y = p.run(x, 2)
    torch.cuda.synchronize()
    p.status()
    ref = torch.from_numpy(oracle.sweep_f64(u0, W, 2)).to(TYPES[dtype][1])
    assert torch.equal(y.cpu(), ref)
    z = x.clone()
    p.run(z, 2, out=z)
    assert torch.equal(z, y)
    p.close()


@pytest.mark.parametrize("dtype,gate", [("bf16", 4e-3), ("f32", 1e-6)])
def test_agrees_with_one_row_kernel(dtype, gate):
    """Random data: the same operands and FP32 accumulation in another order, so
    a last-bit difference of the stored type at most per step."""
    W = inputs.pattern_weights("box49")
    shape = (4100, 4104)
    x = torch.from_numpy(inputs.field(*shape)).cuda().to(TYPES[dtype][1])
    a = _plan(shape, W, dtype).run(x, 2).double()
    b = _plan(shape, W, dtype, phase=False, mma_n=TYPES[dtype][2]).run(x, 2).double()
    assert float((a - b).norm() / b.norm()) <= gate


def test_expired_wait_reports_timeout_and_device_recovers():
    from paper_2605_07954_gb300 import StencilError
    W = np.full((7, 7), 0.125, dtype=np.float32)
    shape = (4096, 4096)
    x = torch.ones(shape, device="cuda", dtype=torch.bfloat16)
    bad = _plan(shape, W, "bf16", timeout_ms=100, debug_withhold=1)
    bad.run(x, 1)
    torch.cuda.synchronize()
    with pytest.raises(StencilError, match="TIMEOUT"):
        bad.status()
    good = _plan(shape, W, "bf16")
    y = good.run(x, 1)
    torch.cuda.synchronize()
    good.status()
    assert float(y[100, 100]) == 6.125
