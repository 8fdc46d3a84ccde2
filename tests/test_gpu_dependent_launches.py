"""Launches that are set up while the kernel before them still runs (small
compactions, batch plans, batched generation): each sees everything before it on
its stream, kernels of the caller and copies too, and they can be captured
behind copies, kernels and joins of other streams."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import ka_inputs as ki  # noqa: E402
import oracle  # noqa: E402
from gpu_util import Workspace, empty, to_dev, to_host, word  # noqa: E402
from test_gpu_batch import GEN, ITEM, table_to_dev  # noqa: E402


@pytest.fixture(scope="module")
def ka(cuda_ok):
    import paper_1709_07781_gb300 as m
    return m


def chain(ka, x, mid, out, counts, ws, n, st):
    """Two dependent compactions: odd population count, then a third of the rest."""
    assert ka.ka_compact(x, n, None, ka.KA_PRED_POPC_ODD, 0, 0, mid, counts, ws.ptr, ws.nbytes, None, st) == 0
    assert ka.ka_compact(mid, n, counts, ka.KA_PRED_MOD_NE0, 3, 0, out, counts[1:], ws.ptr, ws.nbytes, None, st) == 0


def expected(x):
    return oracle.compact(oracle.compact(x, "popc_odd", 0)[0], "mod_ne0", 3)[0]


@pytest.mark.parametrize("n", [1000, 100003, 300001])
def test_between_the_callers_own_kernels(ka, n):
    """The caller's kernels change the input before every pair of calls and
    take the result after it, 60 times without a wait."""
    x = ki.uniform_u32(n, n)
    ws = Workspace(ka, n)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        d_x, mid, out, counts = to_dev(x), empty(n), empty(n), empty(2)
        kept = []
        for i in range(60):
            d_x.add_(1)
            mid.fill_(0)
            chain(ka, d_x, mid, out, counts, ws, n, st)
            kept.append((out.clone(), counts.clone()))
    st.synchronize()
    for i in (0, 1, 17, 58, 59):
        want = expected(x + np.uint32(i + 1))
        o, c = kept[i]
        assert word(c, 1) == want.size and np.array_equal(to_host(o, want.size), want)


@pytest.mark.parametrize("n", [1000, 100003])
def test_captured_behind_copies_and_joins(ka, n):
    x = [ki.uniform_u32(n + i, n) for i in range(3)]
    ws = Workspace(ka, n)
    src, d_x, mid, out, counts, side = to_dev(x[0]), empty(n), empty(n), empty(n), empty(2), empty(n)
    st, other = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(st):  # set-up outside the capture
        d_x.copy_(src)
        chain(ka, d_x, mid, out, counts, ws, n, st)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        d_x.copy_(src)                      # a copy before the first call
        chain(ka, d_x, mid, out, counts, ws, n, st)
        other.wait_stream(st)
        with torch.cuda.stream(other):
            side.copy_(out)                 # a branch
        d_x.copy_(src)
        st.wait_stream(other)               # and its join, two kinds of node before a call
        chain(ka, d_x, mid, out, counts, ws, n, st)
        side.add_(1)
    for xi in x:
        src.copy_(to_dev(xi))
        g.replay()
        torch.cuda.synchronize()
        want = expected(xi)
        assert word(counts, 1) == want.size and np.array_equal(to_host(out, want.size), want)
        assert np.array_equal(to_host(side, want.size), want + np.uint32(1))
    assert ws.status(ka) == 0


def test_generation_and_batches_in_turn(ka):
    """Generation over the same arena before every batch, in place, without a
    wait: each batch reads its own generation."""
    r = np.random.RandomState(3)
    sizes = r.randint(1, 20000, 300)
    off = np.concatenate([[0], np.cumsum((sizes + 3) // 4 * 4)])
    buf, counts = empty(int(off[-1])), empty(sizes.size)
    ws = Workspace(ka, int(sizes.sum()), batch_items=sizes.size)
    st = torch.cuda.Stream()
    t = np.zeros(sizes.size, dtype=ITEM)
    t["in"] = t["out"] = buf.data_ptr() + 4 * off[:-1]
    t["n"], t["pred"], t["param"] = sizes, ka.KA_PRED_POPC_ODD, 0
    t["count"] = counts.data_ptr() + 4 * np.arange(sizes.size)
    gens = []
    for k in range(20):
        g = np.zeros(sizes.size, dtype=GEN)
        g["out"], g["n"], g["seed"] = t["in"], sizes, 1000 * k + np.arange(sizes.size)
        gens.append(table_to_dev(g))
    table = table_to_dev(t)
    torch.cuda.synchronize()
    kept = []
    with torch.cuda.stream(st):
        for k in range(20):
            assert ka.ka_generate_batch(gens[k], sizes.size, sizes.size, ws.ptr, ws.nbytes, st) == 0
            assert ka.ka_compact_batch(table, sizes.size, sizes.size, ws.ptr, ws.nbytes, None, 0, st) == 0
            kept.append((buf.clone(), counts.clone()))
    st.synchronize()
    for k in (0, 7, 19):
        b, c = (to_host(v) for v in kept[k])
        for i in range(0, sizes.size, 23):
            want = oracle.compact(oracle.generate(1000 * k + i, int(sizes[i])), "popc_odd", 0)[0]
            assert c[i] == want.size and np.array_equal(b[off[i]: off[i] + want.size], want), (k, i)
