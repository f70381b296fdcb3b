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


def _grads(u0, W, T, gT, boundary, entry, **opts):
    from paper_2605_07954_gb300 import Plan, _adjoint
    p = Plan(u0.shape[0], u0.shape[1], W, boundary=boundary, **opts)
    gu, gw = _adjoint(p, torch.from_numpy(u0).cuda(), torch.from_numpy(gT).cuda(), T, 0, entry)
    torch.cuda.synchronize()
    p.status()
    p.close()
    return gu.cpu().numpy(), gw.cpu().numpy()


@pytest.mark.parametrize("entry", ["stencil_adjoint", "stencil_adjoint_w32"])
@pytest.mark.parametrize("name", ["heat5", "box9", "star9", "box25", "star13", "box49"])
@pytest.mark.parametrize("boundary", ["zero", "periodic"])
@pytest.mark.parametrize("shape", [(1, 1), (7, 3), (32, 120), (33, 121), (65, 239), (40, 244), (200, 361)])
def test_gradients(oracle, name, boundary, shape, entry):
    W = _weights(name)
    u0 = inputs.field(*shape)
    T = 11
    gT = (inputs.field(*shape, stream=inputs.STREAM_TARGET) - 0.5).astype(np.float32)
    ref_u, ref_w = oracle.adjoint_f64(u0, W, T, gT.astype(np.float64), boundary)
    gu, gw = _grads(u0, W, T, gT, boundary, entry)
    # T steps of `taps` FP32 products each, and their sums over the grid
    assert np.linalg.norm(gu - ref_u) <= 1e-5 * np.linalg.norm(ref_u)
    assert np.linalg.norm(gw - ref_w) <= 1e-5 * np.linalg.norm(ref_w)
    # the states of the streaming kernels have the same bits, so the gradients have
    # (small boxes: cluster-resident kernel)
    tiles = name not in ("box25", "box49") or shape[0] * shape[1] > 20000
    if entry == "stencil_adjoint_w32" and tiles and not (boundary == "periodic" and shape[1] % 4):
        su, sw = _grads(u0, W, T, gT, boundary, entry, kernel="stream")
        assert np.array_equal(gu, su) and np.array_equal(gw, sw)
    assert rel_l2(gu, ref_u) <= 1e-5


@pytest.mark.parametrize("name", ["heat5", "star13"])
@pytest.mark.parametrize("shape,boundary", [((260, 300), "zero"), ((261, 303), "periodic"), ((1003, 1201), "periodic"),
                                            ((1001, 1202), "zero")])
def test_fp64_sums_keep_their_bits(name, shape, boundary):
    """FP64 weight gradients and residuals do not change with the register tiles: a
    default plan gives what the kernel it would otherwise have gives, and is back
    on its own kernel after the call."""
    from paper_2605_07954_gb300 import Plan, StencilError, adjoint
    W = _weights(name)
    x = torch.from_numpy(inputs.field(*shape)).cuda()
    gT = torch.from_numpy(inputs.field(*shape, stream=inputs.STREAM_TARGET) - np.float32(0.5)).cuda()
    try:
        q = Plan(*shape, W, boundary=boundary, kernel="resident")
    except StencilError:
        q = Plan(*shape, W, boundary=boundary, kernel="stream")
    p = Plan(*shape, W, boundary=boundary)
    info, y = p.info(), p.run(x, 9)
    for a, b in zip(adjoint(p, x, gT, 11), adjoint(q, x, gT, 11)):
        assert torch.equal(a, b)
    ra, rb = p.run_residual(x, 23, 5)[1], q.run_residual(x, 23, 5)[1]
    assert np.array_equal(np.asarray(ra.cpu() if hasattr(ra, "cpu") else ra),
                          np.asarray(rb.cpu() if hasattr(rb, "cpu") else rb))
    assert p.info() == info and torch.equal(p.run(x, 9), y)


@pytest.mark.parametrize("name", ["star9", "star13", "box49"])
@pytest.mark.parametrize("boundary,nx", [("zero", 361), ("periodic", 361), ("periodic", 364)])
@pytest.mark.parametrize("col", [117, 119, 120, 122, 239, 240, 355, 360])
def test_an_infinite_lambda_gives_infinite_sums(name, boundary, nx, col):
    """(Grids large enough for the kernel in registers.)  One infinite lambda times positive u: every tap's sum is infinite, not NaN, next
    to the columns where a warp's strip ends and beside the grid's last column too."""
    if boundary == "zero" and col + 3 >= nx:
        col = nx - 4  # (nearer the edge the term u~ = 0 beyond it is 0 x inf)
    W = _weights(name)
    u0 = inputs.field(2800, nx) + np.float32(0.5)
    gT = np.zeros((2800, nx), dtype=np.float32)
    gT[1400, col] = np.inf
    for entry in ("stencil_adjoint_w32", "stencil_adjoint"):
        _, gw = _grads(u0, W, 1, gT, boundary, entry)
        assert np.all(np.isposinf(gw)), entry


@pytest.mark.parametrize("name", ["star9", "star13", "box49"])
def test_sums_beyond_fp32_stay_finite(name):
    """Lambdas of 1e36: the sums of 128 lanes leave the FP32 range, their FP64 sum does not."""
    W = _weights(name)
    u0 = inputs.field(2800, 362) + np.float32(0.5)
    gT = np.full((2800, 362), 1e36, dtype=np.float32)
    _, gw = _grads(u0, W, 1, gT, "periodic", "stencil_adjoint_w32")
    _, ref = _grads(u0, W, 1, gT, "periodic", "stencil_adjoint")
    assert np.all(np.isfinite(gw)) and rel_l2(gw / 1e36, ref / 1e36) <= 1e-5


@pytest.mark.parametrize("entry", ["stencil_adjoint", "stencil_adjoint_w32"])
@pytest.mark.parametrize("T", [1, 2, 3])
@pytest.mark.parametrize("name,shape", [("heat5", (945, 1700)), ("star13", (1000, 1022)), ("box25", (900, 1000))])
def test_few_steps(name, shape, T, entry):
    """One or two recomputed states: the gradients of a streaming plan, bit for bit."""
    W = _weights(name)
    u0 = inputs.field(*shape)
    gT = (inputs.field(*shape, stream=inputs.STREAM_TARGET) - 0.5).astype(np.float32)
    for a, b in zip(_grads(u0, W, T, gT, "zero", entry), _grads(u0, W, T, gT, "zero", entry, kernel="stream")):
        assert np.array_equal(a, b)


# Either side of the sizes from which the reverse step keeps its rows in registers, and
# widths that cut its strips of 120 columns and its chunks of 4.
@pytest.mark.parametrize("name", ["star9", "box25", "star13", "box49"])
@pytest.mark.parametrize("boundary", ["zero", "periodic"])
@pytest.mark.parametrize("shape", [(600, 499), (600, 500), (600, 501), (901, 499), (902, 499), (1000, 501), (1253, 364),
                                   (2779, 361), (8400, 120), (8500, 121)])
def test_gradients_of_larger_grids(oracle, name, boundary, shape):
    W = _weights(name)
    u0 = inputs.field(*shape)
    T = 2
    gT = (inputs.field(*shape, stream=inputs.STREAM_TARGET) - 0.5).astype(np.float32)
    ref_u, ref_w = oracle.adjoint_f64(u0, W, T, gT.astype(np.float64), boundary)
    gu, gw = _grads(u0, W, T, gT, boundary, "stencil_adjoint_w32")
    assert np.linalg.norm(gu - ref_u) <= 1e-5 * np.linalg.norm(ref_u)
    assert np.linalg.norm(gw - ref_w) <= 1e-5 * np.linalg.norm(ref_w)
