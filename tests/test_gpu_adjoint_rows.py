"""GPU tests of the any-width reverse step and of the states that chip-resident
plans recompute in one launch: both gradients against the FP64 oracle at the
edges of the 120-column, 32-row tiles."""
import numpy as np
import pytest

from paper_2605_07954_gb300 import inputs
from _util import rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07954_gb300 import build
    build.build()


def _weights(name):
    if name in ("star9", "box25"):
        return inputs.random_weights("star" if name == "star9" else "box", 2)
    return inputs.pattern_weights(name)


def _grads(u0, W, T, gT, boundary, **opts):
    from paper_2605_07954_gb300 import Plan, adjoint
    p = Plan(u0.shape[0], u0.shape[1], W, boundary=boundary, **opts)
    gu, gw = adjoint(p, torch.from_numpy(u0).cuda(), torch.from_numpy(gT).cuda(), T)
    torch.cuda.synchronize()
    p.status()
    p.close()
    return gu.cpu().numpy(), gw.cpu().numpy()


@pytest.mark.parametrize("name", ["heat5", "box9", "star9", "box25", "star13", "box49"])
@pytest.mark.parametrize("boundary", ["zero", "periodic"])
@pytest.mark.parametrize("shape", [(1, 1), (7, 3), (32, 120), (33, 121), (65, 239), (40, 244), (200, 361)])
def test_gradients(oracle, name, boundary, shape):
    W = _weights(name)
    u0 = inputs.field(*shape)
    T = 11
    gT = (inputs.field(*shape, stream=inputs.STREAM_TARGET) - 0.5).astype(np.float32)
    ref_u, ref_w = oracle.adjoint_f64(u0, W, T, gT.astype(np.float64), boundary)
    gu, gw = _grads(u0, W, T, gT, boundary)
    # T steps of `taps` FP32 products each, and their sums over the grid
    assert np.linalg.norm(gu - ref_u) <= 1e-5 * np.linalg.norm(ref_u)
    assert np.linalg.norm(gw - ref_w) <= 1e-5 * np.linalg.norm(ref_w)
    # the states of the streaming kernels have the same bits, so the gradients have
    if not (boundary == "periodic" and shape[1] % 4):
        su, sw = _grads(u0, W, T, gT, boundary, kernel="stream")
        assert np.array_equal(gu, su) and np.array_equal(gw, sw)
    assert rel_l2(gu, ref_u) <= 1e-5
