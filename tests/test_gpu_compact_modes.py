"""The two ways a block of the fused TMA compaction uses its shared memory (kept
entries moved to a ring per warp, or held in their stage), chosen from the
block's first tile: every density on either side of the choice, data whose
density changes after it, and the edges inside each, bit for bit against the
oracle, in place too."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import ka_inputs as ki  # noqa: E402
import oracle  # noqa: E402
from gpu_util import Workspace, empty, stream, to_dev, to_host, word  # noqa: E402

# entries per tile and resident blocks per SM of each shape's compaction
SHAPES = {(768, 16): (11264, 1), (512, 16): (8192, 2), (256, 16): (4096, 3)}
HALF = 1 << 31  # kept: x < HALF


@pytest.fixture(scope="module")
def ka(cuda_ok):
    import paper_1709_07781_gb300 as m
    return m


def with_density(n, density, seed):
    """n values of which entry i is kept with probability density[i]."""
    u = ki.uniform_f64(seed, n)
    x = ki.uniform_u32(seed + 1, n)
    return np.where(u < density, x >> np.uint32(1), x | np.uint32(HALF)).astype(np.uint32)


def check(ka, x, tile, in_place=False):
    n = x.size
    ws = Workspace(ka, n, tile)
    d_x, d_count = to_dev(x, pad=4), empty(1)
    d_out = d_x if in_place else empty(n + 4)
    assert ka.ka_compact(d_x, n, None, ka.KA_PRED_LT, HALF, 0, d_out, d_count, ws.ptr, ws.nbytes, tile,
                         stream()) == 0
    torch.cuda.synchronize()
    y, k = oracle.compact(x, "lt", HALF)
    assert word(d_count) == k
    assert np.array_equal(to_host(d_out, k), y)
    assert ws.status(ka) == 0


def rounds(tile, r):
    """Entries of r tiles for every resident block."""
    t, per_sm = SHAPES[tile]
    return torch.cuda.get_device_properties(0).multi_processor_count * per_sm * t * r


@pytest.mark.parametrize("tile", sorted(SHAPES))
@pytest.mark.parametrize("s", [0.0, 0.002, 0.02, 0.04, 0.1, 0.15, 0.18, 0.2, 0.6, 1.0])
def test_uniform_density(ka, tile, s):
    n = rounds(tile, 20) + 7
    x = with_density(n, s, 40 + int(100 * s))
    check(ka, x, tile)
    check(ka, x, tile, in_place=True)


@pytest.mark.parametrize("tile", sorted(SHAPES))
@pytest.mark.parametrize("first, rest", [(0.01, 1.0), (0.15, 0.5), (1.0, 0.0), (0.5, 0.01)])
def test_density_that_changes_after_the_first_tiles(ka, tile, first, rest):
    n = rounds(tile, 18) + 3
    density = np.full(n, rest)
    density[: rounds(tile, 1)] = first
    check(ka, with_density(n, density, 61), tile)


@pytest.mark.parametrize("tile", sorted(SHAPES))
def test_density_that_changes_from_segment_to_segment(ka, tile):
    """Sparse first tiles, then segments of 0, 1, 20, 21, 64 and 512 kept
    entries (and between) in random order: rings that fill up, tiles counted
    again, groups of unequal tiles."""
    n = rounds(tile, 16) + 515
    head = rounds(tile, 1)
    per_segment = np.array([0, 1, 20, 21, 64, 100, 300, 512])
    r = np.random.RandomState(5)
    kept = per_segment[r.randint(0, per_segment.size, n // 512 + 1)]
    kept[: head // 512] = 3
    x = ki.uniform_u32(7, n) | np.uint32(HALF)
    place = np.arange(n) % 512
    shift = r.randint(0, 512, kept.size)
    keep = (place + np.repeat(shift, 512)[:n]) % 512 < np.repeat(kept, 512)[:n]
    x[keep] &= np.uint32(HALF - 1)
    check(ka, x, tile)
    check(ka, x, tile, in_place=True)


@pytest.mark.parametrize("n", [11263, 11264, 11265, 2 * 11264 + 1])
@pytest.mark.parametrize("s", [0.01, 0.5])
def test_tile_edges(ka, n, s):
    check(ka, with_density(n, s, n), (768, 16))


@pytest.mark.parametrize("tile", [(128, 4), (256, 4), (128, 16), (512, 8), (1024, 8)])
@pytest.mark.parametrize("off", [0, 1, 3])
def test_arrays_whose_tiles_all_run_at_once(ka, tile, off):
    """The wave kernel of the register shapes: one entry to a full wave and one
    tile past it (the ticketed kernel), inputs at every word of 16 bytes,
    device lengths below the capacity, every predicate kind, in place."""
    t = tile[0] * tile[1]
    wave = torch.cuda.get_device_properties(0).multi_processor_count * (2048 // tile[0])
    for n in (1, t - 1, t, t + 1, 37 * t + 5, min(wave, 1216) * t - off, wave * t + t + 1):
        x = ki.uniform_u32(n & 0xFFF, n)
        buf = to_dev(np.concatenate([np.zeros(off, np.uint32), x]), pad=4)
        for name, param, xform in (("lt", HALF, 0), ("mod_ne0", 12, 1), ("and_mask_eq0", 3, 0), ("popc_odd", 0, 1),
                                   ("ne", int(x[0]), 0), ("lt", 0, 0)):
            for live in (None, n // 2, 0):
                ws = Workspace(ka, n, tile)
                d_out, d_count = empty(n + 4), empty(1)
                d_n = None if live is None else to_dev(np.array([live], np.uint32))
                kind = getattr(ka, "KA_PRED_" + name.upper())
                assert ka.ka_compact(buf.data_ptr() + 4 * off, n, d_n, kind, param, xform, d_out, d_count, ws.ptr,
                                     ws.nbytes, tile, stream()) == 0
                torch.cuda.synchronize()
                want = x if live is None else x[:live]
                y, k = oracle.compact(oracle.map_hash(want) if xform else want, name, param)
                got = to_host(d_out)
                assert word(d_count) == k and ws.status(ka) == 0
                assert np.array_equal(got[:k], y) and (got[k:] == 0xDEADBEEF).all()
        check(ka, x, tile, in_place=True)


@pytest.mark.parametrize("n", [(3 << 17) - 1, 3 << 17, 2490367, 2490369, 3000001, 4980735, 4980737])
@pytest.mark.parametrize("off", [0, 1])
def test_default_kernel_by_size(ka, n, off):
    """Calls without a shape around the sizes where the default kernel changes."""
    x = ki.uniform_u32(n & 0xFFF, n)
    buf = to_dev(np.concatenate([np.zeros(off, np.uint32), x]), pad=4)
    for live in (None, n - 8191):
        ws = Workspace(ka, n)
        d_out, d_count = empty(n + 4), empty(1)
        d_n = None if live is None else to_dev(np.array([live], np.uint32))
        assert ka.ka_compact(buf.data_ptr() + 4 * off, n, d_n, ka.KA_PRED_MOD_NE0, 3, 1, d_out, d_count, ws.ptr,
                             ws.nbytes, None, stream()) == 0
        torch.cuda.synchronize()
        y, k = oracle.compact(oracle.map_hash(x if live is None else x[:live]), "mod_ne0", 3)
        got = to_host(d_out)
        assert word(d_count) == k and ws.status(ka) == 0
        assert np.array_equal(got[:k], y) and (got[k:] == 0xDEADBEEF).all()
    check(ka, x, None, in_place=True)
