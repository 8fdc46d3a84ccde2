"""Inputs of fused runs that a stage refuses on its own: the run refuses them
too."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import ka_inputs as ki  # noqa: E402
from gpu_util import to_dev  # noqa: E402
from test_gpu_actors import compose  # noqa: E402
from test_gpu_fused_runs import ka, spawn_all, system  # noqa: E402,F401


@pytest.mark.parametrize("apart", [False, True])
@pytest.mark.parametrize("n, status", [(5, "KA_E_ARG"), (0, "KA_OK")])
def test_interleave_with_an_array_that_is_not_there(ka, system, n, status, apart):  # noqa: F811
    """Reference to no memory (length 0) as the second array."""
    actors = spawn_all(ka, system, ["prep", ("c", "ne", 0, 0)])
    pipe = compose(ka, *reversed(actors))
    if apart:
        for a in actors:
            assert ka.ka_debug_fail_stage(a, 1 << 30) == 0
    d_x = to_dev(ki.uniform_u32(1, 8))
    _, x = ka.ka_ref_wrap(system, d_x.data_ptr(), n, n)
    _, nothing = ka.ka_ref_wrap(system, 0, 0, 0)
    torch.cuda.synchronize()
    s, q = ka.ka_request(pipe, ka.make_msg([x, nothing]))
    assert s == 0
    s, msg = ka.ka_receive(q)
    assert s == getattr(ka, status) and msg.count == 0
