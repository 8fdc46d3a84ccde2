"""The smallest workspace that a call without a shape takes, asked for again and
again (the answer is kept per thread) and with calls of other sizes and
explicit shapes between: one byte less is refused, before any CUDA call."""
import pytest


@pytest.fixture(scope="module")
def ka():
    import paper_1709_07781_gb300 as m
    return m


def smallest(n, per_tile):
    tiles = -(-n // per_tile)
    return 256 + -(-2 * tiles * 32 // 256) * 256


def refused(ka, n, nbytes, tile=None):
    # addresses that no call touches: the size is refused first
    return ka.ka_compact(0x1000, n, None, ka.KA_PRED_LT, 1, 0, 0x2000, 0x3000, 0x10000, nbytes, tile, None)


@pytest.mark.parametrize("order", [1, -1])
def test_smallest_workspace(ka, order):
    sizes = [(1, 1024), (100003, 1024), ((1 << 21) - 1, 1024), (1 << 21, 2048), (3000001, 2048), ((1 << 22) - 1, 2048),
             (1 << 22, 12288), (1 << 28, 12288)][::order]
    for _ in range(3):
        for n, per_tile in sizes:
            for _ in range(2):
                assert refused(ka, n, smallest(n, per_tile) - 1) == ka.KA_E_WORKSPACE
            assert refused(ka, n, smallest(n, 512) - 1, (128, 4)) == ka.KA_E_WORKSPACE
