"""Runs of stages that the actor layer issues as one kernel: chains of hash maps
and compactions, the flag/scan/move triple, and the interleave in front of
them. Every result equals the oracle's stage-by-stage pipeline, and that of the
same actors issued stage by stage (a failure armed far in the future on the
first stage keeps its run apart)."""
import itertools

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import ka_inputs as ki  # noqa: E402
import oracle  # noqa: E402
from gpu_util import to_dev  # noqa: E402
from test_gpu_actors import compose, result_data, spawn  # noqa: E402


@pytest.fixture(scope="module")
def ka(cuda_ok):
    import paper_1709_07781_gb300 as m
    return m


@pytest.fixture()
def system(ka):
    s, h = ka.ka_system_create(0)
    assert s == 0, ka.ka_strerror(s)
    yield h
    assert ka.ka_system_destroy(h, 1) == 0


# stage kinds of the descriptions below: "prep", "map", ("c", pred, param, hash), ("t", pred, param)
def spawn_all(ka, sys_h, stages, tile=(0, 0)):
    kinds = {p: getattr(ka, "KA_PRED_" + p.upper()) for p in ki.PREDICATES}
    out = []
    for st in stages:
        if st == "prep":
            out.append(spawn(ka, sys_h, ka.KA_STAGE_PREPARE))
        elif st == "map":
            out.append(spawn(ka, sys_h, ka.KA_STAGE_MAP_HASH))
        elif st[0] == "c":
            out.append(spawn(ka, sys_h, ka.KA_STAGE_COMPACT, kinds[st[1]], st[2], st[3], tile))
        else:
            out.append(spawn(ka, sys_h, ka.KA_STAGE_PREDICATE, kinds[st[1]], st[2]))
            out.append(spawn(ka, sys_h, ka.KA_STAGE_EXSCAN))
            out.append(spawn(ka, sys_h, ka.KA_STAGE_SCATTER))
    return out


def expected(arrays, stages):
    x = arrays[0]
    for st in stages:
        if st == "prep":
            x = oracle.prepare_index(arrays[0], arrays[1])
        elif st == "map":
            x = oracle.map_hash(x)
        else:
            if st[0] == "c" and st[3]:
                x = oracle.map_hash(x)
            x, _ = oracle.compact(x, st[1], st[2])
    return x


def request(ka, sys_h, actors, pipe, arrays, offsets):
    dev, refs = [], []
    for x, o in zip(arrays, offsets):
        t = to_dev(np.concatenate([np.zeros(o, np.uint32), x]), pad=4)
        dev.append(t)
        s, r = ka.ka_ref_wrap(sys_h, t.data_ptr() + 4 * o, x.size, x.size)
        assert s == 0
        refs.append(r)
    torch.cuda.synchronize()
    s, q = ka.ka_request(pipe, ka.make_msg(refs))
    assert s == 0
    s, msg = ka.ka_receive(q)
    for r in refs:
        ka.ka_ref_release(r)
    if s != 0:
        return s, None
    y = result_data(ka, msg.refs[0], msg.count)
    ka.ka_ref_release(msg.refs[0])
    return s, y


CHAINS = {
    "pipeline4": ["map", ("c", "topbits_lt", 8, 0), ("c", "popc_odd", 0, 0), ("c", "mod_ne0", 3, 0)],
    "low": [("c", "lt", 1 << 26, 0), ("c", "and_mask_eq0", 1, 0)],  # few kept: the rings
    "hash_each": [("c", "ne", 0, 1), ("c", "lt", 3 << 30, 1), "map"],
    "triple": [("t", "and_mask_eq0", 3)],
    "triple_then": [("t", "popc_odd", 0), ("c", "lt", 1 << 31, 0)],
    # five tests: a run of four, then a run of one stage
    "five": [("c", "lt", 0xF0000000, 0), ("c", "popc_odd", 0, 1), ("c", "ne", 5, 0), "map", ("c", "mod_ne0", 6, 0)],
}
# every set of different tests, and chains that combine or stay chains
KINDS = {"and": ("c", "and_mask_eq0", 1, 0), "lt": ("c", "lt", 0xC0000000, 0), "popc": ("c", "popc_odd", 0, 0),
         "mod": ("c", "mod_ne0", 6, 0), "ne": ("c", "ne", 8, 0)}
for _r in (2, 3, 4):
    for _c in itertools.combinations(sorted(KINDS), _r):
        CHAINS["set " + " ".join(_c)] = [KINDS[k] for k in _c]
CHAINS["set lt and hash"] = ["map", KINDS["lt"], ("c", "lt", 0xE0000000, 0), KINDS["and"]]
CHAINS["one test"] = ["map", ("c", "lt", 1 << 31, 0), ("c", "lt", 1 << 30, 0)]
CHAINS["everything"] = ["map", ("c", "lt", 0xFFFFFFFF, 0), "map"]
CHAINS["two divisors"] = [KINDS["mod"], ("c", "mod_ne0", 5, 0)]
CHAINS["two values"] = [KINDS["ne"], ("c", "ne", 9, 0)]
# edges of segments, of both tile sizes (8192 and 11264 entries), of one round
# of every resident block, and several rounds
SIZES = [1, 3, 511, 513, 8191, 8193, 11263, 11265, 304 * 8192 + 5, (1 << 22) + 1, 152 * 11264 * 9 + 7]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("name", sorted(CHAINS))
def test_chain_of_one_array(ka, system, name, n):
    stages = CHAINS[name]
    actors = spawn_all(ka, system, stages)
    pipe = compose(ka, *reversed(actors))
    x = ki.uniform_u32(n & 0xFFFF, n)
    want = expected([x], stages)
    for offset in (0, 1, 3):
        s, got = request(ka, system, actors, pipe, [x], [offset])
        assert s == 0 and np.array_equal(got, want)
    assert ka.ka_debug_fail_stage(actors[0], 1 << 30) == 0
    s, apart = request(ka, system, actors, pipe, [x], [0])
    assert s == 0 and np.array_equal(apart, want)


INTERLEAVED = {
    "zeros": ["prep", ("c", "ne", 0, 0)],
    "triple": ["prep", ("t", "ne", 0)],
    "chain": ["prep", ("c", "ne", 0, 1), ("c", "popc_odd", 0, 0)],
}


@pytest.mark.parametrize("k", [1, 2, 255, 257, 4095, 4097, 5631, 5633, 304 * 4096 + 3, 152 * 5632 * 5 + 1])
@pytest.mark.parametrize("zero", [0.0, 0.5, 0.99])
def test_chain_of_an_interleave(ka, system, zero, k):
    a, b = ki.index_pairs(k, zero, seed=k & 0xFFF)
    for name, stages in sorted(INTERLEAVED.items()):
        actors = spawn_all(ka, system, stages)
        pipe = compose(ka, *reversed(actors))
        want = expected([a, b], stages)
        # 16-byte aligned arrays share a kernel; others are interleaved first
        for offsets in ((0, 0), (4, 0), (1, 0), (2, 2)):
            s, got = request(ka, system, actors, pipe, [a, b], offsets)
            assert s == 0 and np.array_equal(got, want), (name, offsets)


@pytest.mark.parametrize("tile", [(256, 4), (512, 16), (768, 16)])
def test_live_length_from_an_earlier_stage(ka, system, tile):
    """A stage with a tile of its own runs alone; the run after it reads its
    length from the device, as does a chain after a chain."""
    n = (1 << 22) + 17
    x = ki.uniform_u32(9, n)
    head, tail = [("c", "lt", 1 << 31, 0)], [("c", "popc_odd", 0, 1), ("c", "mod_ne0", 3, 0)]
    actors = spawn_all(ka, system, head, tile) + spawn_all(ka, system, tail)
    pipe = compose(ka, *reversed(actors))
    s, got = request(ka, system, actors, pipe, [x], [0])
    assert s == 0 and np.array_equal(got, expected([x], head + tail))


def test_an_actor_twice_in_a_run(ka, system):
    x = ki.uniform_u32(10, 70001)
    a = spawn_all(ka, system, [("c", "popc_odd", 0, 1)])[0]
    pipe = compose(ka, a, a, a)
    s, got = request(ka, system, [a], pipe, [x], [0])
    assert s == 0 and np.array_equal(got, expected([x], [("c", "popc_odd", 0, 1)] * 3))


def test_injected_failure_inside_a_run(ka, system):
    """An armed stage counts its own messages: the first passes, the second fails."""
    x = ki.uniform_u32(11, 5000)
    actors = spawn_all(ka, system, CHAINS["pipeline4"])
    pipe = compose(ka, *reversed(actors))
    assert ka.ka_debug_fail_stage(actors[2], 1) == 0
    assert request(ka, system, actors, pipe, [x], [0])[0] == 0
    assert request(ka, system, actors, pipe, [x], [0])[0] == ka.KA_E_INJECTED
    assert ka.ka_debug_fail_stage(actors[2], -1) == 0
    assert request(ka, system, actors, pipe, [x], [0])[0] == 0


@pytest.mark.parametrize("name, outputs", [("pipeline4", 2), ("triple", 3), ("triple_then", 3)])
def test_budget_of_a_run_is_that_of_its_stages(ka, name, outputs):
    """The budget admits what it admits stage by stage: the most outputs alive
    at once, with one byte less refused on both paths."""
    n = 100000
    block = (4 * n + 255) // 256 * 256 + 256
    x = ki.uniform_u32(12, n)
    for spare, status in ((0, ka.KA_OK), (-1, ka.KA_E_BUDGET)):
        for apart in (False, True):
            s, sys_h = ka.ka_system_create(0, budget_bytes=outputs * block + spare)
            assert s == 0
            actors = spawn_all(ka, sys_h, CHAINS[name])
            pipe = compose(ka, *reversed(actors))
            if apart:
                assert ka.ka_debug_fail_stage(actors[0], 1 << 30) == 0
                assert ka.ka_debug_fail_stage(actors[-1], 1 << 30) == 0
            assert request(ka, sys_h, actors, pipe, [x], [0])[0] == status, (spare, apart)
            assert ka.ka_system_destroy(sys_h, 1) == 0
