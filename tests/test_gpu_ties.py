"""Coincident geometry: pixels where several triangles have the same depth key.  Every copy of a visible
triangle is visible, however many there are.  Bits, compared exactly.
"""
import numpy as np
import pytest

from test_gpu_large import View, join, quad
from test_gpu_parity import F  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def test_four_billion_ties(F):  # noqa: F811
    """257 copies of a quad that covers 4,096 x 4,096 pixels: 256 ties a pixel, 2^32 in all."""
    n, W = 257, 4096
    mesh = join([quad([(-2, -2, 0.25), (2, -2, 0.25), (2, 2, 0.25), (-2, 2, 0.25)])] * n)
    v = View(F, mesh, np.eye(4, dtype=np.float32), W, W)
    bits = v.bits()
    v.close()
    assert int(np.unpackbits(bits.view(np.uint8)).sum()) == 2 * n
