"""Pixels that the paired orbit does not take (near the tip of the set, |c|^2 above
3.6, and imaginary parts below 2^-90): two at a time by the definition's
operations, bit for bit against the oracle."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_mandelbrot_pairs import check, ka  # noqa: E402,F401

TIP = (-1.98, -0.02, -1.90, 0.02)
# (nan corners make no pixel finite: every step is taken)
VIEWS = [TIP, (-1.945, -0.003, -1.938, 0.003), (-1.9856, -0.0004, -1.985, 0.0004), (-2.0, -1e-6, -1.99999, 1e-6),
         (-1.99, -1e-30, -1.9, 1e-30), (-1.3, 1e-30, 0.2, 2e-30), (-1e38, -1e38, 1e38, 1e38),
         (float("nan"), -1.0, 1.0, 1.0)]


@pytest.mark.parametrize("rect", VIEWS)
@pytest.mark.parametrize("iters", [0, 1, 2, 9, 1000])
def test_views(ka, rect, iters):  # noqa: F811
    check(ka, 61, 43, rect, iters)
    check(ka, 64, 3, rect, iters, offset=1)


@pytest.mark.parametrize("w, h", [(1, 1), (2, 1), (1, 3), (3, 3), (257, 1)])
def test_odd_sizes(ka, w, h):  # noqa: F811
    check(ka, w, h, TIP, 300)
