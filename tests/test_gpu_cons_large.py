"""Conservative marking of large hidden triangles, clipped ones too: their boxes are shared by the grid as tiles.
Bits against the oracle, compared exactly; times against the second rasterization in the same process.
"""
import numpy as np
import pytest

from test_gpu_large import View, forward, grounds, join, patch, walls
from test_gpu_parity import F  # noqa: F401  (fixture)
from test_gpu_ties import reference

pytestmark = pytest.mark.gpu

FRONT = patch(64, 3.0, -2.0)


def slivers(n, seed=9):
    """Long thin triangles: boxes of every shape, many without a sample, some past the window."""
    rng = np.random.default_rng(seed)
    a = rng.uniform(-1.3, 1.3, (n, 2))
    ang, ln = rng.uniform(0, 2 * np.pi, n), 2.0 ** rng.uniform(-8, 1, n)
    ang[::4] = 0.0  # along a row
    d = np.stack([np.cos(ang), np.sin(ang)], 1) * ln[:, None]
    w = np.stack([-d[:, 1], d[:, 0]], 1) / ln[:, None] * (2.0 ** rng.uniform(-11, -4, n))[:, None]
    z = rng.uniform(-0.9, 0.9, (n, 1, 1)) + rng.uniform(-0.05, 0.05, (n, 3, 1))
    pos = np.concatenate([np.stack([a, a + d, a + 0.5 * d + w], 1), z], 2).reshape(-1, 3).astype(np.float32)
    return pos, np.arange(3 * n, dtype=np.uint32).reshape(-1, 3)


SCENES = {
    "ground_behind": lambda: (join([FRONT, grounds(1)]), None, 640, 360),
    "walls_behind": lambda: (join([FRONT, walls(6)]), None, 640, 360),
    "both_in_front": lambda: (join([walls(2), grounds(2, y=-0.5), patch(200, 5.0, -6.0, 3)]), None, 501, 333),
    "slivers": lambda: (slivers(3000), np.eye(4, dtype=np.float32), 700, 410),
    "few_slivers": lambda: (slivers(40), np.eye(4, dtype=np.float32), 700, 410),
    "sliver_window": lambda: (slivers(3000), np.eye(4, dtype=np.float32), 1024, 3),
}


@pytest.mark.parametrize("name", sorted(SCENES))
def test_conservative_large(F, name):  # noqa: F811
    import torch
    (pos, idx), M, W, H = SCENES[name]()
    M = forward(W, H) if M is None else M
    want = reference(M, pos, idx, W, H, True)
    v = View(F, (pos, idx), M, W, H)
    assert want.any() and (v.bits(F.FA_VIS_CONSERVATIVE) == want).all()
    dm = torch.as_tensor(np.asarray(M, np.float32).reshape(16)).cuda()
    for flags in (0, F.FA_FRAME_PERSISTENT):
        bufs = F.FrameBuffers.allocate(len(idx), len(pos), 16)
        F.atlas_frame_dev_matrix(v.ctx, v.mesh, bufs, dm, W, H, 1.0, 10, flags=flags | F.FA_VIS_CONSERVATIVE)
        torch.cuda.synchronize()
        assert (bufs.vt.cpu().numpy().view(np.uint32) == want).all()
        v.ctx.device_status()  # (more charts than the context has room for: not what is asked here)
    v.close()


@pytest.mark.parametrize("mesh", [lambda: grounds(1), lambda: walls(1), lambda: grounds(20)],
                         ids=["ground", "wall", "grounds"])
def test_conservative_large_time(F, mesh):  # noqa: F811
    """Behind a mesh that fills the view: no slower than two rasterizations (half as much again is left for the
    clock's steps)."""
    W, H = 960, 540
    v = View(F, join([FRONT, mesh()]), forward(W, H), W, H)
    one, two = v.ms(F.FA_VIS_CONSERVATIVE, reps=10), v.ms(F.FA_VIS_CONSERVATIVE, F.FA_RASTER_HIZ, reps=10)
    v.close()
    assert one <= 1.5 * two, (one, two)
