"""GPU tests of the chip-resident register-tile kernel (AUTO plans of grids that
fit the chip as one tile per SM).

It computes the same products in the same order as the kernel it stands in for
(the cluster-resident one where the grid fits it, else the streaming one), so
FP32 results are compared bit for bit (streaming kernel, periodic widths that are not a multiple
of 4: to FP32 rounding, as for the streaming kernel's own depths); 16-bit
storage is rounded only at the end, so its results are the rounded FP32 ones.
"""
import numpy as np
import pytest

from paper_2605_07954_gb300 import inputs
from _util import fp32_tol, rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TDT = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


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


def _plan(shape, W, grid=True, **kw):
    from paper_2605_07954_gb300 import Plan
    p = Plan(shape[0], shape[1], W, **kw)
    if grid and not (W.shape[0] >= 5 and np.count_nonzero(W) > 13 and shape[0] * shape[1] <= 20000):  # (cluster-resident)
        i = p.info()
        assert i["kernel"] == 6 and i["ctas"] == 1 and i["halo_cols"] % 4 == 0, i
    return p


def _reference_plan(shape, W, boundary="zero"):
    """The cluster-resident kernel where the grid fits it, else the streaming kernel."""
    from paper_2605_07954_gb300 import StencilError
    try:
        return _plan(shape, W, grid=False, boundary=boundary, kernel="resident")
    except StencilError:
        return _plan(shape, W, grid=False, boundary=boundary, kernel="stream")


# One tile, one strip, one tile row, chunks and warps cut by the grid's edge,
# widths around the 128 staged columns, and about the largest grids that fit.
SHAPES = [(1, 1), (2, 3), (1, 700), (700, 1), (127, 128), (33, 129), (130, 517), (301, 252), (512, 512),
          (1000, 1022), (1201, 1100)]


@pytest.mark.parametrize("boundary", ["zero", "periodic"])
@pytest.mark.parametrize("name", ["heat5", "box9", "star9", "box25", "star13", "box49"])
@pytest.mark.parametrize("shape", SHAPES)
def test_same_bits_as_the_kernel_it_stands_in_for(name, shape, boundary):
    W = _weights(name)
    x = torch.from_numpy(inputs.field(*shape)).cuda()
    p = _plan(shape, W, boundary=boundary)
    q = _reference_plan(shape, W, boundary)
    for T in (1, 2, 7, 33):
        y, z = p.run(x, T), q.run(x, T)
        torch.cuda.synchronize()
        p.status()
        if boundary == "periodic" and shape[1] % 4 and q.info()["kernel"] == 2:
            assert rel_l2(y.cpu().numpy(), z.cpu().numpy().astype(np.float64)) <= fp32_tol(T), T
        else:
            assert torch.equal(y, z), T
    p.close()
    q.close()


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("shape", [(200, 336), (131, 333)])
def test_16_bit_storage_rounds_once(dtype, shape):
    W = inputs.pattern_weights("box9")
    x = torch.from_numpy(inputs.field(*shape)).cuda().to(TDT[dtype])
    y = _plan(shape, W, dtype=dtype).run(x, 40)
    z = _reference_plan(shape, W).run(x.float(), 40)
    assert torch.equal(y, z.to(TDT[dtype]))


@pytest.mark.parametrize("T", [1, 2, 3, 9, 40])
@pytest.mark.parametrize("boundary", ["zero", "periodic"])
def test_in_place(T, boundary):
    W = inputs.pattern_weights("star13")
    p = _plan((300, 420), W, boundary=boundary)
    x = torch.from_numpy(inputs.field(300, 420)).cuda()
    z = x.clone()
    y = p.run(x, T)
    p.run(z, T, out=z)
    assert torch.equal(y, z)


def test_unaligned_buffers():
    W = inputs.pattern_weights("box9")
    p = _plan((64, 256), W)
    f = torch.from_numpy(inputs.field(64, 256)).cuda()
    buf = torch.empty(64 * 256 + 1, device="cuda")
    x = buf[1:].view(64, 256)
    x.copy_(f)
    assert torch.equal(p.run(x, 13), p.run(f, 13))


def test_replayed_graph_and_two_streams():
    """Epochs count on from one launch to the next: a captured run replayed
    several times, and two plans running on two streams at once."""
    W = inputs.pattern_weights("heat5")
    p, q = _plan((512, 512), W), _plan((400, 600), W)
    x, y = torch.from_numpy(inputs.field(512, 512)).cuda(), torch.from_numpy(inputs.field(400, 600)).cuda()
    want_x, want_y = p.run(x, 50), q.run(y, 70)
    out = torch.empty_like(x)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s1):
        p.run(x, 50, out=out)
    for _ in range(5):
        out.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(s1):
            g.replay()
        with torch.cuda.stream(s2):
            got_y = q.run(y, 70)
        torch.cuda.synchronize()
        assert torch.equal(out, want_x) and torch.equal(got_y, want_y)
    p.status()
    q.status()


def test_expired_wait_reports_timeout_and_plan_recovers():
    from paper_2605_07954_gb300 import StencilError
    W = inputs.pattern_weights("heat5")
    x = torch.from_numpy(inputs.field(512, 512)).cuda()
    bad = _plan((512, 512), W, timeout_ms=100, debug_withhold=1)
    bad.run(x, 60)
    torch.cuda.synchronize()
    with pytest.raises(StencilError, match="TIMEOUT"):
        bad.status()
    bad.run(x, 1)  # no exchange: nothing to wait for
    bad.status()
    good = _plan((512, 512), W)
    ref = _reference_plan((512, 512), W)
    assert torch.equal(good.run(x, 60), ref.run(x, 60))
    good.status()


# Grids beyond one tile per SM: launches of up to tb_depth steps over two or more
# waves of tiles.  Just above that limit, two waves, tall and wide, ragged.
TILE_SHAPES = [("heat5", (1600, 1600)), ("heat5", (3203, 1021)), ("box9", (1601, 1701)), ("star9", (2048, 2048)),
               ("star9", (1024, 4099)), ("box25", (2001, 2003)), ("star13", (1801, 1804)), ("star13", (8190, 517)),
               ("box49", (2048, 2048)), ("box49", (1701, 1601))]


@pytest.mark.parametrize("boundary", ["zero", "periodic"])
@pytest.mark.parametrize("name,shape", TILE_SHAPES)
def test_launches_of_tiles_same_bits(name, shape, boundary):
    W = _weights(name)
    x = torch.from_numpy(inputs.field(*shape)).cuda()
    p = _plan(shape, W, grid=False, boundary=boundary)
    q = _plan(shape, W, grid=False, boundary=boundary, kernel="stream")
    i = p.info()
    assert i["kernel"] == 2 and i["threads"] > 256 and i["tb_depth"] >= 2, i  # (the streaming kernel: at most 256)
    k = i["tb_depth"]
    for T in (1, 2, k, k + 1, 2 * k + 3):
        y, z = p.run(x, T), q.run(x, T)
        v = x.clone()
        p.run(v, T, out=v)
        if boundary == "periodic" and shape[1] % 4:
            assert rel_l2(y.cpu().numpy(), z.cpu().numpy().astype(np.float64)) <= fp32_tol(T), T
            assert rel_l2(v.cpu().numpy(), z.cpu().numpy().astype(np.float64)) <= fp32_tol(T), T
        else:
            assert torch.equal(y, z) and torch.equal(v, z), T
        assert p.launches(T) == -(-T // k)
    p.close()
    q.close()


@pytest.mark.parametrize("dtype", ["bf16", "f16"])
@pytest.mark.parametrize("name,shape", [("star13", (2048, 2048)), ("heat5", (1000, 1022)), ("box9", (1601, 1701))])
def test_16_bit_storage_keeps_the_streaming_roundings(dtype, name, shape):
    """Grids beyond the cluster-resident kernel: rounded after every launch of the streaming kernel."""
    W = _weights(name)
    x = torch.from_numpy(inputs.field(*shape)).cuda().to(TDT[dtype])
    p = _plan(shape, W, grid=False, dtype=dtype)
    q = _plan(shape, W, grid=False, dtype=dtype, kernel="stream")
    assert p.info()["kernel"] == 2 and torch.equal(p.run(x, 45), q.run(x, 45))


def test_launches_of_tiles_autotuned():
    """Autotuning times the tiles against the streaming kernel's variants; the bits are the same."""
    shape, W = (1801, 1804), inputs.pattern_weights("star13")
    x = torch.from_numpy(inputs.field(*shape)).cuda()
    y = _plan(shape, W, grid=False, autotune=True).run(x, 23)
    again = _plan(shape, W, grid=False, autotune=True)  # (the cached choice)
    z = _plan(shape, W, grid=False, kernel="stream").run(x, 23)
    assert torch.equal(y, z) and torch.equal(again.run(x, 23), z)


# Either side of the lines up to which short runs, and runs of periodic ragged widths,
# take the cluster-resident kernel from a register-tile plan.
CLUSTER_SHAPES = [(140, 141), (141, 142), (180, 200), (181, 200), (100, 200), (101, 200), (60, 249), (250, 251),
                  (255, 257), (50, 201), (50, 199), (250, 112), (251, 112)]


@pytest.mark.parametrize("boundary", ["zero", "periodic"])
@pytest.mark.parametrize("name", ["heat5", "box9", "star9", "box25", "star13", "box49"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_runs_in_one_cluster_have_the_same_bits(name, boundary, dtype):
    """One plan's runs of different lengths may take either kernel: the cluster-resident
    kernel's bits every time, in place as well."""
    W = _weights(name)
    for shape in CLUSTER_SHAPES:
        x = torch.from_numpy(inputs.field(*shape)).cuda().to(TDT[dtype])
        p = _plan(shape, W, grid=False, boundary=boundary, dtype=dtype)
        a = _plan(shape, W, grid=False, boundary=boundary, dtype=dtype, autotune=True)
        q = _plan(shape, W, grid=False, boundary=boundary, dtype=dtype, kernel="resident")
        for T in (1, 2, 1, 3, 4, 25, 1):
            want = q.run(x, T)
            z = x.clone()
            p.run(z, T, out=z)
            assert torch.equal(p.run(x, T), want) and torch.equal(z, want), (shape, T)
        assert torch.equal(p.run(p.run(x, 1), 1), q.run(q.run(x, 1), 1))
        for T in (1, 2, 25):
            y = a.run(x, T)
            if a.info()["kernel"] == 6:  # (autotuning may keep the streaming kernel, whose bits differ)
                assert torch.equal(y, q.run(x, T)), (shape, T)
        p.status()
        for plan in (p, a, q):
            plan.close()


@pytest.mark.parametrize("boundary", ["zero", "periodic"])
@pytest.mark.parametrize("name,shape", [("heat5", (1833, 1459)), ("heat5", (1600, 1600)), ("box9", (1601, 1701)),
                                        ("star9", (2047, 1801)), ("box25", (1800, 2047)), ("star13", (1801, 1804)),
                                        ("star13", (1800, 2047)), ("box49", (1701, 1601))])
def test_short_launches_of_tile_plans_have_the_same_bits(name, shape, boundary):
    """Runs of up to a few steps, and the remainders of longer ones, stream: every count
    from 1 to one past a launch of tiles, in and out of place."""
    W = _weights(name)
    x = torch.from_numpy(inputs.field(*shape)).cuda()
    p = _plan(shape, W, grid=False, boundary=boundary)
    q = _plan(shape, W, grid=False, boundary=boundary, kernel="stream")
    k = p.info()["tb_depth"]
    want = x
    for T in range(1, min(k, 12) + 2):
        z = x.clone()
        p.run(z, T, out=z)
        y = p.run(x, T)
        if boundary == "periodic" and shape[1] % 4:
            want = q.run(x, T).double()
            for v in (y, z):
                assert float((v.double() - want).norm() / want.norm()) <= fp32_tol(T), T
        else:
            want = q.run(want, 1)
            assert torch.equal(y, want) and torch.equal(z, want), T
    p.close()
    q.close()
