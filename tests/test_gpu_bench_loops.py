"""The benchmark's direct loop with and without stages that share a kernel: the
lengths that the same stages give as a composite, at both waits."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import ka_inputs as ki  # noqa: E402
from gpu_util import to_dev  # noqa: E402
from test_gpu_fused_runs import CHAINS, expected, ka  # noqa: E402,F401


def specs_of(ka, stages):
    kinds = {p: getattr(ka, "KA_PRED_" + p.upper()) for p in ki.PREDICATES}
    out = []
    for st in stages:
        if st == "prep":
            out.append((ka.KA_STAGE_PREPARE, 0, 0, 0))
        elif st == "map":
            out.append((ka.KA_STAGE_MAP_HASH, 0, 0, 0))
        elif st[0] == "c":
            out.append((ka.KA_STAGE_COMPACT, kinds[st[1]], st[2], st[3]))
        else:
            out += [(ka.KA_STAGE_PREDICATE, kinds[st[1]], st[2], 0), (ka.KA_STAGE_EXSCAN, 0, 0, 0),
                    (ka.KA_STAGE_SCATTER, 0, 0, 0)]
    return out


@pytest.mark.parametrize("n", [1, 70001, (1 << 22) + 3])
@pytest.mark.parametrize("name", ["pipeline4", "triple", "triple_then", "five", "everything"])
def test_lengths(ka, name, n):  # noqa: F811
    x = ki.uniform_u32(n & 0xFF, n)
    d_x = to_dev(x)
    torch.cuda.synchronize()
    want = expected([x], CHAINS[name]).size
    for flags in (0, ka.KA_BENCH_WAIT_TAG, ka.KA_BENCH_SHARED, ka.KA_BENCH_WAIT_TAG | ka.KA_BENCH_SHARED):
        s, _, k = ka.ka_bench_direct_chain(specs_of(ka, CHAINS[name]), d_x, n, 2, None, flags)
        assert s == 0 and k == want, flags


@pytest.mark.parametrize("k", [4, 200000, 1 << 21])
def test_lengths_behind_an_interleave(ka, k):  # noqa: F811
    import numpy as np
    a, b = ki.index_pairs(k, 0.5, seed=k & 0xFFF)
    d = to_dev(np.concatenate([a, b]))
    torch.cuda.synchronize()
    stages = ["prep", ("t", "ne", 0), ("c", "popc_odd", 0, 1)]
    want = expected([a, b], stages).size
    for flags in (0, ka.KA_BENCH_SHARED):
        s, _, got = ka.ka_bench_direct_chain(specs_of(ka, stages), d, k, 2, None, flags)
        assert s == 0 and got == want, flags
