"""GPU tests of the batched path: many grids in one persistent, graph-replayed launch.

Every grid of a batch must give exactly the bits of a single-grid stencil_run
(the arithmetic per point does not depend on tiling or depth), and match the
FP64 oracle within the FP32 gate.  The 256-grid workload (sides log-uniform
in [64, 2048], half Heat-5pt and half Box-9pt with random normalised weights,
200 steps) runs in full.
"""
import numpy as np
import pytest

from paper_2605_07954_gb300 import inputs
from _util import fp32_tol, rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07954_gb300 import build
    build.build()


def _single(x, W, T, boundary):
    # the batch runs the streaming kernel's arithmetic, so compare with that kernel
    # (small grids would otherwise get the cluster-resident kernel's summation order)
    from paper_2605_07954_gb300 import Plan
    p = Plan(x.shape[0], x.shape[1], W, boundary=boundary, kernel="stream")
    y = p.run(x, T)
    torch.cuda.synchronize()
    p.close()
    return y


def _mixed_grids():
    """Ragged widths, odd heights, tiny and multi-tile grids, T not a multiple of k."""
    rng = np.random.default_rng(31)
    shapes = [(64, 64), (67, 203), (300, 517), (129, 1000), (5, 7), (1, 33), (600, 600),
              (40, 2100), (257, 96), (33, 1), (800, 130), (2, 2)]
    grids = []
    for i, (ny, nx) in enumerate(shapes):
        kind = ["heat5r", "box9", "star13", "box49"][i % 4]
        if kind in ("heat5r", "box9"):
            W = inputs.batch_grid_weights(kind, i)
        else:
            W = inputs.pattern_weights(kind, stream=2000 + i)
        boundary = "periodic" if (i % 3 == 2 and nx % 4 == 0) else "zero"
        T = int(rng.integers(0, 40))
        x = torch.from_numpy(inputs.field(ny, nx, stream=500 + i)).cuda()
        grids.append(dict(x=x, out=torch.empty_like(x), weights=W, T=T, boundary=boundary))
    return grids


@pytest.mark.parametrize("tb_depth,threads", [(0, 0), (2, 64), (4, 256), (1, 128)])
def test_mixed_batch_bitwise_equals_single_runs(oracle, tb_depth, threads):
    from paper_2605_07954_gb300 import Batch
    grids = _mixed_grids()
    b = Batch(grids, tb_depth=tb_depth, threads=threads, tile_rows=(0 if tb_depth else 48))
    b.run()
    torch.cuda.synchronize()
    b.status()
    info = b.info()
    assert info["n"] == len(grids) and info["launches"] >= 1
    for i, g in enumerate(grids):
        ref = _single(g["x"], g["weights"], g["T"], g["boundary"])
        assert torch.equal(g["out"], ref), (i, g["x"].shape, g["T"], info)
        if g["x"].numel() <= 300 * 600:
            want = oracle.sweep_f64(g["x"].cpu().numpy(), g["weights"], g["T"], g["boundary"])
            assert rel_l2(g["out"].cpu().numpy(), want) <= fp32_tol(g["T"]), i
    # the graph replays: a second run gives the same bits
    first = [g["out"].clone() for g in grids]
    b.run()
    torch.cuda.synchronize()
    for g, f in zip(grids, first):
        assert torch.equal(g["out"], f)
    b.close()


def test_in_place_grids():
    from paper_2605_07954_gb300 import Batch
    W = inputs.batch_grid_weights("box9", 3)
    x = torch.from_numpy(inputs.field(333, 444)).cuda()
    ref = _single(x, W, 25, "zero")
    z = x.clone()
    b = Batch([dict(x=z, out=z, weights=W, T=25)])
    b.run()
    torch.cuda.synchronize()
    assert torch.equal(z, ref)
    b.close()


def test_withheld_item_times_out_and_reports():
    """A work item whose completion is never published: the dependent waits run
    out after timeout_ms, the kernel returns, and the status word says TIMEOUT."""
    from paper_2605_07954_gb300 import Batch, StencilError
    W = inputs.batch_grid_weights("box9", 1)
    x = torch.from_numpy(inputs.field(1024, 1024)).cuda()
    g = [dict(x=x, out=torch.empty_like(x), weights=W, T=64)]
    b = Batch(g, tb_depth=8, timeout_ms=200, debug_withhold_item=1)
    b.run()
    torch.cuda.synchronize()
    with pytest.raises(StencilError, match="TIMEOUT"):
        b.status()
    b.close()
    # the device is healthy afterwards: a normal batch runs and is correct
    b2 = Batch(g, tb_depth=8)
    b2.run()
    torch.cuda.synchronize()
    b2.status()
    assert torch.equal(g[0]["out"], _single(x, W, 64, "zero"))
    b2.close()


def _workload_256():
    sides, kinds = inputs.batch_spec(256)
    grids = []
    for gi, (s, kind) in enumerate(zip(sides, kinds)):
        W = inputs.batch_grid_weights(kind, gi)
        x = torch.from_numpy(inputs.field(int(s), int(s), stream=10000 + gi)).cuda()
        grids.append(dict(x=x, out=torch.empty_like(x), weights=W, T=200))
    return grids


def test_batched_256_grids_workload(oracle):
    """The 256-grid, 200-step batch: every grid bit-equal to its single-grid run;
    the smallest grids also against the FP64 oracle; maximum principle on all."""
    from paper_2605_07954_gb300 import Batch
    grids = _workload_256()
    b = Batch(grids)
    b.run()
    torch.cuda.synchronize()
    b.status()
    order = sorted(range(len(grids)), key=lambda i: grids[i]["x"].shape[0])
    for i in range(len(grids)):
        g = grids[i]
        out = g["out"]
        assert float(out.min()) >= 0.0 and float(out.max()) <= float(g["x"].max()) * (1 + 1e-5)
        if i % 8 == 0 or i in order[:4] or i in order[-2:]:
            assert torch.equal(out, _single(g["x"], g["weights"], 200, "zero")), i
    for i in order[:3]:
        g = grids[i]
        want = oracle.sweep_f64(g["x"].cpu().numpy(), g["weights"], 200)
        assert rel_l2(g["out"].cpu().numpy(), want) <= fp32_tol(200)
    b.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_one_warp_tiles_edges_and_queues(dtype):
    """Radius-1 grids run as one-warp tiles from two queues (boxes, stars): widths
    around a tile's 112 and 120 columns, chunks cut by the right edge, periodic
    grids of several tiles, heights around the tile heights; with one queue empty
    too.  Against single runs: FP32 bit for bit, BF16 within its rounding (the
    two round after different numbers of steps)."""
    from paper_2605_07954_gb300 import Batch
    td = torch.float32 if dtype == "f32" else torch.bfloat16
    shapes = [(300, 111), (97, 121), (33, 240), (129, 226), (64, 1025), (700, 5), (512, 480), (31, 112)]
    for kinds in (("heat5r", "box9"), ("heat5r",), ("box9",)):
        for depth in (0, 8, 1):
            grids = []
            for i, (ny, nx) in enumerate(shapes):
                x = torch.from_numpy(inputs.field(ny, nx, stream=700 + i)).cuda().to(td)
                grids.append(dict(x=x, out=torch.empty_like(x), T=17 + i, boundary="periodic" if nx % 16 == 0 else "zero",
                                  weights=inputs.batch_grid_weights(kinds[i % len(kinds)], i)))
            b = Batch(grids, dtype=dtype, tb_depth=depth, tile_rows=0 if depth != 8 else 40)
            assert b.info()["threads"] == 32
            for _ in range(2):
                b.run()
            torch.cuda.synchronize()
            b.status()
            for i, g in enumerate(grids):
                if dtype == "f32":
                    assert torch.equal(g["out"], _single(g["x"], g["weights"], g["T"], g["boundary"])), (kinds, depth, i)
                else:
                    ref = _single(g["x"].float(), g["weights"], g["T"], g["boundary"]).double()
                    err = float((g["out"].double() - ref).norm() / ref.norm())
                    assert err <= 2.0 ** -8, (kinds, depth, i, err)
            b.close()


@pytest.mark.parametrize("name", ["box9", "star13", "box49"])
def test_periodic_grids_of_many_tiles(name):
    """Periodic grids wrap, so a tile at one edge also waits for the tiles at the
    opposite one: many small tiles, several runs, CTA-wide tiles (threads set)."""
    from paper_2605_07954_gb300 import Batch
    W = inputs.pattern_weights(name)
    grids = []
    for i, (ny, nx) in enumerate([(400, 1036), (1001, 260), (260, 2100)]):
        x = torch.from_numpy(inputs.field(ny, nx, stream=900 + i)).cuda()
        grids.append(dict(x=x, out=torch.empty_like(x), weights=W, T=24, boundary="periodic"))
    b = Batch(grids, threads=64, tile_rows=24)
    for _ in range(3):
        b.run()
        torch.cuda.synchronize()
        b.status()
        for i, g in enumerate(grids):
            assert torch.equal(g["out"], _single(g["x"], W, 24, "periodic")), i
    b.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
def test_one_warp_tiles_read_what_their_neighbours_wrote(dtype):
    """Many low one-warp tiles, each block of steps reading rows that up to eight
    other SMs wrote in the block before: every run has the bits of a streaming
    plan that rounds after the same 8 steps (16-bit rows are read through L1)."""
    from paper_2605_07954_gb300 import Batch, Plan
    td = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}[dtype]
    grids, want = [], []
    for i, (ny, nx, kind) in enumerate([(1200, 1000, "box9"), (1500, 340, "heat5r"), (900, 2048, "heat5r"),
                                        (333, 777, "box9")]):
        W = inputs.batch_grid_weights(kind, i)
        x = torch.from_numpy(inputs.field(ny, nx, stream=40 + i)).cuda().to(td)
        grids.append(dict(x=x, out=torch.empty_like(x), weights=W, T=160))
        p = Plan(ny, nx, W, dtype=dtype, kernel="stream", tb_depth=8, threads=128)
        want.append(p.run(x, 160))
        torch.cuda.synchronize()
        p.close()
    b = Batch(grids, dtype=dtype, tb_depth=8, tile_rows=12)
    assert b.info()["threads"] == 32
    for _ in range(10):
        for g in grids:
            g["out"].zero_()
        b.run()
        torch.cuda.synchronize()
        b.status()
        assert all(torch.equal(g["out"], w) for g, w in zip(grids, want))
    b.close()
