"""GPU tests of the one-warp streaming kernel of large radius-1 plans: the bits of
the CTA-wide kernel at widths the right edge cuts, both boundaries, and the three
storage types (same launches, so the same roundings)."""
import pytest

from paper_2605_07954_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TDT = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07954_gb300 import build
    build.build()


# (4 or 8 columns per lane for the star) x (aligned, a chunk cut after 4, padded rows)
@pytest.mark.parametrize("name", ["heat5", "box9"])
@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("shape,boundary", [((4104, 4096), "zero"), ((4096, 4100), "periodic"), ((3700, 4099), "zero"),
                                            ((6600, 7012), "zero"), ((6600, 7013), "zero"), ((6600, 7012), "periodic")])
def test_same_bits_as_cta_wide_kernel(name, dtype, shape, boundary):
    from paper_2605_07954_gb300 import Plan
    W = inputs.pattern_weights(name)
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    x = torch.rand(shape, generator=g, device="cuda").to(TDT[dtype])
    p = Plan(shape[0], shape[1], W, dtype=dtype, boundary=boundary)
    q = Plan(shape[0], shape[1], W, dtype=dtype, boundary=boundary, threads=128 if name == "heat5" else 64)
    assert p.info()["threads"] == 32 and p.info()["tb_depth"] == q.info()["tb_depth"] == 8
    for T in (8, 19):
        y = p.run(x, T)
        assert torch.equal(y, q.run(x, T)), T
        z = x.clone()
        p.run(z, T, out=z)
        # in place, an odd number of launches is cut otherwise, which 16-bit storage sees
        if dtype == "f32":
            assert torch.equal(z, y), T
    p.close()
    q.close()


@pytest.mark.parametrize("nx,columns", [(8192, 8), (8188, 4), (8191, 4), (8190, 4)])
def test_wide_chunks_only_where_no_chunk_is_cut(nx, columns):
    """8 columns a lane for the 5-point star on widths that are a multiple of 8, else 4
    (tiles of at most 240 and 112 columns); the bits of the CTA-wide kernel either way."""
    from paper_2605_07954_gb300 import Plan
    W = inputs.pattern_weights("heat5")
    g = torch.Generator(device="cuda")
    g.manual_seed(6)
    x = torch.rand((8190, nx), generator=g, device="cuda")
    p, q = Plan(8190, nx, W), Plan(8190, nx, W, threads=128)
    i = p.info()
    assert i["threads"] == 32 and (112 < i["tile_cols"] <= 240) == (columns == 8), i
    assert torch.equal(p.run(x, 17), q.run(x, 17))
    p.close()
    q.close()


@pytest.mark.parametrize("name", ["heat5", "box9"])
@pytest.mark.parametrize("ny,nx", [(7192, 2000), (7050, 2000), (7186, 2001), (4100, 4096), (4096, 4372),
                                   (8192, 8180), (8000, 2020), (8000, 1801)])
def test_the_last_tiles_are_large_enough(name, ny, nx):
    """Tile sizes that would leave a last row of tiles lower than the 11 rows, or a last
    strip narrower than the 8 columns, that the tiles beside them read beyond their own
    are changed; the bits are the CTA-wide kernel's."""
    from paper_2605_07954_gb300 import Plan
    W = inputs.pattern_weights(name)
    g = torch.Generator(device="cuda")
    g.manual_seed(9)
    x = torch.rand((ny, nx), generator=g, device="cuda")
    p, q = Plan(ny, nx, W), Plan(ny, nx, W, threads=128 if name == "heat5" else 64)
    i = p.info()
    assert i["threads"] == 32 and (ny % i["tile_rows"] == 0 or ny % i["tile_rows"] >= 11), i
    assert nx % i["tile_cols"] == 0 or nx % i["tile_cols"] >= 8, i
    assert torch.equal(p.run(x, 17), q.run(x, 17))
    p.close()
    q.close()
