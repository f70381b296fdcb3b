"""Periodic convergence checks (stencil_run_residual): residuals ||u_t - u_{t-1}||_2
after every m-th step against the FP64 oracle, and the final state bit-identical
to stencil_run."""
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


@pytest.mark.parametrize("name,boundary", [("box9", "zero"), ("star13", "periodic"), ("heat5", "zero")])
@pytest.mark.parametrize("T,m", [(23, 5), (10, 1), (4, 9), (24, 8)])
def test_residuals_match_oracle(oracle, name, boundary, T, m):
    from paper_2605_07954_gb300 import Plan
    W = inputs.pattern_weights(name)
    # periodic widths that are multiples of 4 keep results independent of the
    # launch depths (see test_depth_does_not_change_bits)
    nx = 256 if boundary == "periodic" else 257
    u0 = inputs.field(130, nx)
    p = Plan(130, nx, W, boundary=boundary)
    x = torch.from_numpy(u0).cuda()
    y, res = p.run_residual(x, T, m)
    ref_final = p.run(x, T)
    torch.cuda.synchronize()
    assert torch.equal(y, ref_final)
    assert res.numel() == T // m
    states = [u0.astype(np.float64)]
    for t in range(T):
        states.append(oracle.sweep_f64(states[-1], W, 1, boundary))
    want = [np.linalg.norm(states[t] - states[t - 1]) for t in range(m, T + 1, m)]
    np.testing.assert_allclose(res.cpu().numpy(), want, rtol=2e-4)
    p.close()


def test_fullsize_residuals_nonincreasing():
    """8192^2 Box-9 (non-negative weights summing to 1, zero boundary): the
    step operator is a contraction, so the residual never grows."""
    from paper_2605_07954_gb300 import Plan
    W = inputs.pattern_weights("box9")
    p = Plan(8192, 8192, W)
    x = torch.from_numpy(inputs.field(8192, 8192)).cuda()
    y, res = p.run_residual(x, 1000, 100)
    ref = p.run(x, 1000)
    torch.cuda.synchronize()
    assert torch.equal(y, ref)
    r = res.cpu().numpy()
    assert len(r) == 10 and np.all(r > 0)
    assert np.all(r[1:] <= r[:-1] * (1 + 1e-6))
    p.close()


@pytest.mark.parametrize("name,shape,boundary", [("box9", (1700, 1600), "zero"), ("heat5", (1604, 1800), "periodic"),
                                                 ("star13", (1600, 1504), "zero"), ("box49", (1600, 1504), "periodic"),
                                                 ("box9", (300, 333), "zero"), ("star13", (300, 332), "periodic")])
@pytest.mark.parametrize("m", [1, 2, 3, 6, 8, 9, 13])
def test_last_two_steps_of_every_interval(name, shape, boundary, m):
    """Intervals whose last launch stores two steps (streaming and chip-resident
    plans), single steps and remainders: the final state has the bits of a plain
    run, and every residual is that of the states two runs give."""
    from paper_2605_07954_gb300 import Plan
    W = inputs.pattern_weights(name)
    x = torch.from_numpy(inputs.field(*shape)).cuda()
    p = Plan(shape[0], shape[1], W, boundary=boundary)
    T = 3 * m + 1
    for _ in range(2):
        y, res = p.run_residual(x, T, m)
        p.status()
        assert torch.equal(y, p.run(x, T))
        want = [torch.linalg.vector_norm(p.run(x, t).double() - p.run(x, t - 1).double()) for t in range(m, T + 1, m)]
        # FP64 sums of exact differences: rounding at 45 bits and better
        assert torch.allclose(res, torch.stack(want), rtol=1e-11, atol=0)
    p.close()


@pytest.mark.parametrize("scale", [1e-30, 1e25, float("inf")])
def test_residual_outside_the_fp32_range(scale):
    """Differences whose squares leave the FP32 range, and infinities."""
    from paper_2605_07954_gb300 import Plan
    W = inputs.pattern_weights("box9")
    x = torch.from_numpy(inputs.field(60, 68)).cuda() * (scale if scale < 1e30 else 1.0)
    if scale == float("inf"):
        x[3, 5] = scale
    p = Plan(60, 68, W)
    _, res = p.run_residual(x, 4, 2)
    want = [torch.linalg.vector_norm(p.run(x, t).double() - p.run(x, t - 1).double()) for t in (2, 4)]
    assert torch.allclose(res, torch.stack(want), rtol=1e-11, atol=0, equal_nan=True)
    p.close()


@pytest.mark.parametrize("side", [1024, 16384])
def test_large_differences_keep_a_finite_sum(side):
    """Differences near 1e18: on the larger grid a thread adds about a thousand
    squares of 1e36 each, more than FP32 holds."""
    from paper_2605_07954_gb300 import Plan
    W = np.zeros((3, 3), dtype=np.float32)
    W[1, 1] = 2.0  # u_1 - u_0 = u_0
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    x = torch.rand((side, side), generator=g, device="cuda").add_(0.5).mul_(2.0 ** 59)
    p = Plan(side, side, W)
    _, res = p.run_residual(x, 1, 1)
    want = torch.linalg.vector_norm(x, dtype=torch.float64)
    # two FP64 sums of positive terms (at most 2^-53 per addition, fewer than 2000 in a row)
    assert torch.allclose(res[0], want, rtol=2e-13, atol=0)
    p.close()


def test_sum_is_as_accurate_as_fp64():
    """Differences that need more than 24 bits, against their exact sum: 16 terms per
    thread, then some 20 additions of FP64 numbers one after the other."""
    from paper_2605_07954_gb300 import Plan
    W = np.zeros((3, 3), dtype=np.float32)
    W[1, 1] = 2.0 ** -13  # u_0 - u_1 = u_0 (1 - 2^-13), 37 bits
    n = np.random.default_rng(1).integers(1 << 23, 1 << 24, size=(2048, 2048))
    p = Plan(2048, 2048, W)
    _, res = p.run_residual(torch.from_numpy(n.astype(np.float32)).cuda(), 1, 1)
    rows = (n.astype(np.uint64) ** 2).reshape(-1, 4096).sum(axis=1, dtype=np.uint64)  # (each below 2^60)
    exact = sum(int(r) for r in rows) * 8191 ** 2  # x 2^-26
    got = float(res[0].cpu())
    # the square root halves the error of the sum and adds a rounding of its own
    assert abs(got ** 2 * 2.0 ** 26 / exact - 1.0) <= 24 * 2.0 ** -53
    p.close()
