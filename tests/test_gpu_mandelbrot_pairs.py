"""The Mandelbrot kernel's pairs of pixels against the oracle, bit for bit: step
limits around its tested head and runs, odd widths and pixel counts, an output
at an odd word, and rectangles on either side of what the paired orbit takes
(|c|^2 to 3.6, imaginary parts of 0 and below 2^-90)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from gpu_util import empty, stream, to_host  # noqa: E402

WHOLE = (-2.0, -1.25, 0.5, 1.25)


@pytest.fixture(scope="module")
def ka(cuda_ok):
    import paper_1709_07781_gb300 as m
    return m


def check(ka, w, h, rect, iters, offset=0):
    out = empty(w * h + offset + 1)
    assert ka.ka_mandelbrot(out.data_ptr() + 4 * offset, w, h, *rect, iters, stream()) == 0
    torch.cuda.synchronize()
    got = to_host(out)
    assert np.array_equal(got[offset: offset + w * h].reshape(h, w), oracle.mandelbrot(w, h, *rect, iters))
    assert got[-1] == 0xDEADBEEF and (offset == 0 or got[0] == 0xDEADBEEF)


@pytest.mark.parametrize("iters", [0, 1, 4, 7, 8, 9, 11, 12, 13, 16, 50, 203])
def test_step_limits(ka, iters):
    check(ka, 97, 61, WHOLE, iters)
    check(ka, 96, 61, oracle.MANDELBROT_REGION, iters, offset=1)


@pytest.mark.parametrize("w, h", [(1, 1), (1, 2), (2, 1), (3, 3), (1, 257), (255, 1), (257, 5)])
def test_odd_sizes(ka, w, h):
    check(ka, w, h, WHOLE, 100)
    check(ka, w, h, WHOLE, 100, offset=1)


@pytest.mark.parametrize("rect", [
    (-2.1, -0.1, -1.8, 0.1),          # the tip: |c|^2 on both sides of 3.6
    (-3.0, -3.0, 3.0, 3.0),
    (5.0, 5.0, 1e20, 1e20),
    (-1.5, -1e-26, 0.3, 1e-26),       # imaginary parts around 2^-90, and 0
    (-1.5, -1e-37, 0.3, 1e-37),
    (-1.5, 0.0, 0.3, 1e-44),
    (-1e-30, -1.5, 1e-30, 1.5),
])
def test_rectangles(ka, rect):
    check(ka, 64, 48, rect, 300)
