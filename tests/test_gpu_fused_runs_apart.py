"""Composed stages issued one by one (a failure armed far in the future on every
one of them, so that no two of them share a kernel), and the same stages as fused
runs: the same results, budgets and failures."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import ka_inputs as ki  # noqa: E402
from test_gpu_actors import compose  # noqa: E402
from test_gpu_fused_runs import CHAINS, INTERLEAVED, expected, ka, request, spawn_all, system  # noqa: E402,F401


def arm(ka, actors, on=True):
    for a in set(actors):
        assert ka.ka_debug_fail_stage(a, 1 << 30 if on else -1) == 0


@pytest.mark.parametrize("n", [1, 513, 8193, 400009, (1 << 22) + 1])
@pytest.mark.parametrize("name", sorted(CHAINS))
def test_one_array(ka, system, name, n):  # noqa: F811
    stages = CHAINS[name]
    actors = spawn_all(ka, system, stages)
    pipe = compose(ka, *reversed(actors))
    x = ki.uniform_u32(n & 0xFFFF, n)
    want = expected([x], stages)
    for one_by_one in (True, False):
        arm(ka, actors, one_by_one)
        s, got = request(ka, system, actors, pipe, [x], [1])
        assert s == 0 and np.array_equal(got, want), one_by_one


@pytest.mark.parametrize("k", [1, 257, 5633, 200003])
@pytest.mark.parametrize("name", sorted(INTERLEAVED))
def test_interleave(ka, system, name, k):  # noqa: F811
    a, b = ki.index_pairs(k, 0.5, seed=k & 0xFFF)
    actors = spawn_all(ka, system, INTERLEAVED[name])
    pipe = compose(ka, *reversed(actors))
    want = expected([a, b], INTERLEAVED[name])
    for one_by_one in (True, False):
        arm(ka, actors, one_by_one)
        s, got = request(ka, system, actors, pipe, [a, b], [0, 0])
        assert s == 0 and np.array_equal(got, want), one_by_one


# the most outputs of the run that are alive at once, each of n entries
@pytest.mark.parametrize("name, outputs", [("pipeline4", 2), ("triple", 3), ("triple_then", 3), ("five", 2),
                                           ("set and lt popc", 2)])
def test_budget(ka, name, outputs):  # noqa: F811
    n = 100000
    block = (4 * n + 255) // 256 * 256 + 256
    x = ki.uniform_u32(12, n)
    for spare, status in ((0, "KA_OK"), (-1, "KA_E_BUDGET")):
        for one_by_one in (True, False):
            s, sys_h = ka.ka_system_create(0, budget_bytes=outputs * block + spare)
            assert s == 0
            actors = spawn_all(ka, sys_h, CHAINS[name])
            pipe = compose(ka, *reversed(actors))
            arm(ka, actors, one_by_one)
            assert request(ka, sys_h, actors, pipe, [x], [0])[0] == getattr(ka, status), (spare, one_by_one)
            assert ka.ka_system_destroy(sys_h, 1) == 0
