"""Runs of composed stages on either side of the size from which only runs that
kernels are made for are fused: a product between tests, tests that do not
combine, a product after the tests, and runs that go on after them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import ka_inputs as ki  # noqa: E402
from test_gpu_actors import compose  # noqa: E402
from test_gpu_fused_runs import expected, ka, request, spawn_all, system  # noqa: E402,F401

LT = ("c", "lt", 1 << 29, 0)
CHAINS = {
    "product between": [LT, ("c", "popc_odd", 0, 1), ("c", "mod_ne0", 3, 1)],
    "two divisors": ["map", ("c", "mod_ne0", 6, 0), ("c", "mod_ne0", 5, 0), ("c", "popc_odd", 0, 0)],
    "product after": [LT, "map", "map"],
    "product first": ["map", LT, ("c", "popc_odd", 0, 0), "map"],
    "triple and product": [("t", "and_mask_eq0", 3), ("c", "lt", 1 << 31, 1), ("c", "ne", 7, 0)],
}


@pytest.mark.parametrize("n", [(1 << 25) - 1, 1 << 25, (1 << 25) + 12345])
@pytest.mark.parametrize("name", sorted(CHAINS))
def test_around_the_size(ka, system, name, n):  # noqa: F811
    stages = CHAINS[name]
    actors = spawn_all(ka, system, stages)
    pipe = compose(ka, *reversed(actors))
    x = ki.uniform_u32(n & 0xFF, n)
    want = expected([x], stages)
    for offset in (0, 3):
        s, got = request(ka, system, actors, pipe, [x], [offset])
        assert s == 0 and np.array_equal(got, want)
