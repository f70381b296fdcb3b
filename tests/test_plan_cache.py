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
