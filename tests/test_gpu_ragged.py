"""GPU tests of streaming runs on widths that are not a multiple of 4 (padded rows)."""
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


def _weights(name):
    if name in ("star9", "box25"):
        return inputs.random_weights("star" if name == "star9" else "box", 2)
    return inputs.pattern_weights(name)


@pytest.mark.parametrize("name", ["heat5", "box9", "star9", "box25", "star13", "box49"])
@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("shape", [(70, 517), (45, 1030), (300, 1999), (9, 5), (130, 1)])
def test_ragged_widths_through_padded_rows(name, dtype, shape):
    """Streaming runs of several launches on widths that are not a multiple of 4
    go through padded rows: the bits of runs that do not (single launches of the
    same depths on the dense grid), in place as well."""
    from paper_2605_07954_gb300 import Plan
    W = _weights(name)
    x = torch.from_numpy(inputs.field(*shape)).cuda().to(TDT[dtype])
    p = Plan(shape[0], shape[1], W, dtype=dtype, kernel="stream")
    k = p.info()["tb_depth"]
    for T in (2 * k, 3 * k + 1):
        want, t = x, 0
        while t < T:
            want = p.run(want, min(k, T - t))
            t += k
        z = x.clone()
        y = p.run(x, T)
        p.run(z, T, out=z)
        assert torch.equal(y, want) and torch.equal(z, want), T
    p.close()
