"""Coincident geometry: pixels where several triangles have the same depth key.  Every copy of a visible
triangle is visible, however many there are.  Bits, compared exactly.
"""
import numpy as np
import pytest

import oracle as O
from paper_2502_17712_gb300 import scenes as S
from test_gpu_large import View, forward, grounds, join, patch, quad, walls
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


def reference(M, pos, idx, W, H, conservative):
    """The oracle's bits less the triangles outside one side plane: the front end drops those first, and
    conservative marking does not see one that lies within half a snapping step (1/512 pixel) of the window and
    snaps onto its edge, which the oracle counts (no copy of the code before this test ever did)."""
    want = O.visibility(M, pos, idx, W, H, conservative=conservative)
    c = O.transform(M, pos)[idx]
    x, y, w = c[..., 0], c[..., 1], c[..., 3]
    out = (x > w).all(1) | (x < -w).all(1) | (y > w).all(1) | (y < -w).all(1)
    return want & ~O.bool_to_vt(out)


def copies(mesh, n):
    return join([mesh] * n)


# (mesh, matrix, window): small, mid-size and large boxes, clipped fans, many triangles in a small window
OVERFLOWING = {
    "small": lambda: (copies(patch(300, 1.0, 0.0), 3), S.view_proj((0.1, -0.2, 2.2), (0, 0, 0), (0, 1, 0), 500, 400), 500, 400),
    "mid_size": lambda: (copies(patch(40, 3.0, -2.0), 8), forward(400, 300), 400, 300),
    "large": lambda: (copies(walls(2), 8), forward(320, 200), 320, 200),
    "clipped": lambda: (copies(grounds(2), 8), forward(640, 360), 640, 360),
    "behind": lambda: (join([patch(40, 3.0, -2.0), copies(walls(3), 4), copies(patch(200, 5.0, -3.0, 4), 9),
                             copies(patch(150, 0.8, -1.5, 5), 9)]), forward(480, 270), 480, 270),
    "small_window": lambda: (copies(patch(150, 0.5, -1.0), 40), forward(96, 64), 96, 64),
}


@pytest.mark.parametrize("name", sorted(OVERFLOWING))
def test_more_ties_than_lists_hold(F, name):  # noqa: F811
    """Against the oracle, with and without conservative marking, and in one persistent launch."""
    import torch
    (pos, idx), M, W, H = OVERFLOWING[name]()
    v = View(F, (pos, idx), M, W, H)
    for flags in (0, F.FA_VIS_CONSERVATIVE):
        want = reference(M, pos, idx, W, H, bool(flags))
        assert want.any() and (v.bits(flags) == want).all()
        bufs = F.FrameBuffers.allocate(len(idx), len(pos), 16)
        F.atlas_frame(v.ctx, v.mesh, bufs, M, W, H, 1.0, 10, flags=flags | F.FA_FRAME_PERSISTENT)
        torch.cuda.synchronize()
        assert (bufs.vt.cpu().numpy().view(np.uint32) == want).all()
        v.ctx.device_status()  # (more charts than the context has room for: not what is asked here)
    v.close()


@pytest.mark.parametrize("n,radius,k", [(64, 3.0, 2), (64, 3.0, 8), (200, 2.2, 4), (20, 2.0, 8)])
def test_coincident_time(F, n, radius, k):  # noqa: F811
    """k copies of a patch: about as fast as two rasterizations, which know no ties."""
    W, H = 1920, 1080
    sc = S.grid_scene(3, n)
    v = View(F, copies((sc.pos, sc.idx), k), S.view_proj((0.1, -0.2, radius), (0, 0, 0), (0, 1, 0), W, H), W, H)
    one, two = v.ms(reps=20), v.ms(raster=F.FA_RASTER_HIZ, reps=20)
    v.close()
    assert one <= 1.5 * two, (one, two)
