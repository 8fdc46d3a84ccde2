"""Blocks of the fused compaction that start on dense data and go over to rings where
it thins out: changes at every tile of the first laps, back to dense data, at the
ends of arrays and before a ragged tile, in every kernel that does it (one
test, a set, a chain, an interleave), bit for bit against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import ka_inputs as ki  # noqa: E402
import oracle  # noqa: E402
from gpu_util import Workspace, empty, stream, to_dev, to_host, word  # noqa: E402
from test_gpu_compact_modes import HALF, check, ka, with_density  # noqa: E402,F401
from test_gpu_fused_runs import expected, request, spawn_all, system  # noqa: E402,F401
from test_gpu_actors import compose  # noqa: E402

TILE = (768, 16)
T = 11264


def by_round(densities, extra=0):
    """Keep-probabilities: densities[r] for the r-th tile of every resident block."""
    per = torch.cuda.get_device_properties(0).multi_processor_count * T
    return np.concatenate([np.repeat(np.array(densities), per), np.full(extra, densities[-1])])


@pytest.mark.parametrize("dense", [1, 2, 3, 4, 5, 6, 8, 10, 11])
@pytest.mark.parametrize("thin", [0.0, 0.02])
def test_dense_then_thin(ka, dense, thin):  # noqa: F811
    for more in (1, 3, 7):
        for extra in (0, 5, 3 * T + 513):
            d = by_round([0.7] * dense + [thin] * more, extra)
            x = with_density(d.size, d, 3 + dense + more)
            check(ka, x, TILE, in_place=extra == 5)


@pytest.mark.parametrize("pattern", [[1.0] * 3 + [0.0] * 9 + [1.0] * 4, [0.3] * 6 + [0.1] * 12 + [0.9],
                                     [1.0, 0.0] * 9, [0.0, 1.0, 0.02] * 6, [0.5] * 4 + [0.124, 0.126] * 7,
                                     [0.9] * 2 + [0.01] * 5 + [0.2] * 5 + [0.001] * 5])
def test_patterns(ka, pattern):  # noqa: F811
    d = by_round(pattern, 11)
    x = with_density(d.size, d, 17)
    check(ka, x, TILE)
    check(ka, x, TILE, in_place=True)


def test_a_look_back_that_gives_up(ka):  # noqa: F811
    """One poll, then no more: blocks whose look-back gives up still count, change
    over and end; the next call in the same workspace, cleared, is right."""
    d = by_round([0.8] * 4 + [0.01] * 12, 9)
    x = with_density(d.size, d, 41)
    ws = Workspace(ka, x.size, TILE)
    d_x, d_out, d_count = to_dev(x, pad=4), empty(x.size + 4), empty(1)

    def call():
        assert ka.ka_compact(d_x, x.size, None, ka.KA_PRED_LT, HALF, 0, d_out, d_count, ws.ptr, ws.nbytes, TILE,
                             stream()) == 0
        torch.cuda.synchronize()
        return ws.status(ka)

    assert ka.ka_workspace_set_spin_limit(ws.ptr, 1, stream()) == 0
    for _ in range(3):
        assert call() in (0, ka.KA_E_DEVICE_TIMEOUT)
    assert ka.ka_workspace_init(ws.ptr, ws.nbytes, stream()) == 0
    assert call() == 0
    y, k = oracle.compact(x, "lt", HALF)
    assert word(d_count) == k and np.array_equal(to_host(d_out, k), y)


RUNS = {
    "set": [("c", "lt", HALF, 0), ("c", "popc_odd", 0, 0)],
    "chain": [("c", "lt", HALF, 0), ("c", "popc_odd", 0, 1)],
}


@pytest.mark.parametrize("name", sorted(RUNS))
@pytest.mark.parametrize("dense", [2, 5, 7])
def test_fused_runs(ka, system, name, dense):  # noqa: F811
    d = by_round([1.0] * dense + [0.01] * 8, 7)
    x = with_density(d.size, d, 23)
    actors = spawn_all(ka, system, RUNS[name])
    pipe = compose(ka, *reversed(actors))
    s, got = request(ka, system, actors, pipe, [x], [0])
    assert s == 0 and np.array_equal(got, expected([x], RUNS[name]))


@pytest.mark.parametrize("dense", [2, 5, 7])
def test_interleave(ka, system, dense):  # noqa: F811
    d = by_round([0.8] * dense + [0.01] * 8, 8)
    k = d.size // 2
    a, b = (np.where(ki.uniform_f64(29 + i, k) < d[: 2 * k: 2], ki.uniform_u32(31 + i, k) | np.uint32(1), 0)
            .astype(np.uint32) for i in range(2))
    stages = ["prep", ("c", "ne", 0, 0)]
    actors = spawn_all(ka, system, stages)
    pipe = compose(ka, *reversed(actors))
    s, got = request(ka, system, actors, pipe, [a, b], [0, 0])
    assert s == 0 and np.array_equal(got, expected([a, b], stages))
