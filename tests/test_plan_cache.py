"""StencilFn's plan cache, without a GPU: plans are stand-ins that record what happens to them."""
import gc

import numpy as np
import pytest

import paper_2605_07954_gb300 as lib


class FakePlan:
    def __init__(self, ny, nx, W, boundary="zero"):
        self.shape, self.W, self.closed = (ny, nx), W, False

    def set_weights(self, W):
        self.W = W

    def close(self):
        self.closed = True


@pytest.fixture
def cache(monkeypatch):
    monkeypatch.setattr(lib, "Plan", FakePlan)
    return lib._PlanCache(size=3)


W3 = np.ones((3, 3), dtype=np.float32)


def test_a_dropped_plan_stays_usable_for_its_holders(cache):
    """A plan that falls out of the cache between a forward and its backward pass
    belongs to the backward pass until that is done."""
    held = cache.get(0, 10, 10, W3, "zero")
    for n in range(20, 24):
        cache.get(0, n, n, W3, "zero")
    assert len(cache.plans) == 3 and held not in cache.plans.values()
    gc.collect()
    assert not held.closed


def test_every_stream_has_its_own_plans(cache):
    """A plan's launches share its workspace and exchange grids, so two streams never share a plan."""
    a = cache.get(0, 10, 10, W3, "zero", stream=1)
    b = cache.get(0, 10, 10, W3, "zero", stream=2)
    assert a is not b
    assert cache.get(0, 10, 10, W3, "zero", stream=1) is a
    assert cache.get(0, 10, 10, W3, "periodic", stream=2) is not b
    # one stream's many shapes do not push out another's
    for n in range(20, 30):
        cache.get(0, n, n, W3, "zero", stream=2)
    assert cache.get(0, 10, 10, W3, "zero", stream=1) is a
    assert len(cache.plans) == 1 + 3
    # and many streams are bounded as well
    for s in range(3, 40):
        cache.get(0, 10, 10, W3, "zero", stream=s)
    assert len(cache.plans) == 4 * 3


def test_a_captured_call_allocates_nothing(cache):
    """A call under capture takes over the plan that a warm-up on another stream made."""
    a = cache.get(0, 10, 10, W3, "zero", stream=1)
    assert cache.get(0, 10, 10, W3, "zero", stream=9, capturing=lambda: True) is a
    assert cache.get(0, 10, 10, W3, "zero", stream=9) is a
    assert cache.get(0, 10, 10, W3, "zero", stream=1) is not a
