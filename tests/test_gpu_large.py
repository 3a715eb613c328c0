"""Views of few large triangles: sub-triangles that fill the window, many more of their 16x16 tiles than the
tile table has room for, and more of them than there are queue records.  Visible bits against the oracle,
compared exactly; times against the second rasterization (the tile-depth option) in the same process.
"""
import numpy as np
import pytest

import oracle as O
from paper_2502_17712_gb300 import scenes as S
from test_gpu_parity import F  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def quad(p):
    return np.array(p, np.float32), np.array([[0, 1, 2], [0, 2, 3]], np.uint32)


def join(meshes):
    pos, idx, n = [], [], 0
    for p, i in meshes:
        pos.append(p)
        idx.append(i + np.uint32(n))
        n += len(p)
    return np.concatenate(pos), np.concatenate(idx)


def walls(n, seed=1):
    """Walls that fill the view of a camera at the origin looking down -z, tilted a little."""
    rng = np.random.default_rng(seed)
    out = []
    for k in range(n):
        z = -4.0 - 0.1 * k
        d = rng.uniform(-0.2, 0.2, 4)
        out.append(quad([(2 * z, z, z + d[0]), (-2 * z, z, z + d[1]), (-2 * z, -z, z + d[2]), (2 * z, -z, z + d[3])]))
    return join(out)


def grounds(n, y=-1.0, step=0.02):
    """Ground quads below the camera that reach from behind it to z = -100: clipped by the near plane and the
    guard band."""
    return join([quad([(-50, y - step * k, 10), (50, y - step * k, 10), (50, y - step * k, -100),
                       (-50, y - step * k, -100)]) for k in range(n)])


def patch(n, half, z, seed=2):
    """An n x n patch facing the camera."""
    rng = np.random.default_rng(seed)
    x, y = np.meshgrid(np.linspace(-half, half, n), np.linspace(-half, half, n))
    pos = np.stack([x, y, z + rng.uniform(-0.01, 0.01, x.shape)], -1).reshape(-1, 3).astype(np.float32)
    a = (np.arange(n - 1)[None, :] + n * np.arange(n - 1)[:, None]).reshape(-1)
    idx = np.concatenate([np.stack([a, a + 1, a + n], 1), np.stack([a + 1, a + n + 1, a + n], 1)])
    return pos, idx.astype(np.uint32)


def forward(W, H):
    return S.view_proj((0, 0, 0), (0, 0, -1), (0, 1, 0), W, H)


class View:
    def __init__(self, F, mesh, M, W, H):  # noqa: F811
        import torch
        self.F, (pos, idx), self.M, self.W, self.H = F, mesh, M, W, H
        self.ctx = F.Context(max_tris=len(idx), max_verts=len(pos), max_charts=16, max_width=W, max_height=H)
        self.mesh = F.Mesh(self.ctx, pos, idx)
        self.vt = torch.zeros((len(idx) + 31) // 32, dtype=torch.int32, device="cuda")

    def run(self, flags=0, raster=0):
        self.ctx.set_raster_schedule(16, raster)
        self.F.fa_visibility(self.ctx.handle, self.mesh.handle, self.M, self.W, self.H, self.vt, flags=flags)

    def bits(self, flags=0, raster=0):
        import torch
        self.run(flags, raster)
        torch.cuda.synchronize()
        assert self.ctx.device_status() == self.F.FA_OK
        return self.vt.cpu().numpy().view(np.uint32)

    def ms(self, flags=0, raster=0, reps=3):
        import torch
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        best = float("inf")
        self.run(flags, raster)
        for _ in range(reps):
            torch.cuda.synchronize()
            e[0].record()
            self.run(flags, raster)
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        return best

    def close(self):
        self.mesh.close()
        self.ctx.close()


@pytest.fixture
def view(F):  # noqa: F811
    made = []

    def make(*a):
        made.append(View(F, *a))
        return made[-1]

    yield make
    for v in made:
        v.close()


SCENES = {
    "walls": lambda: walls(20),  # 40 triangles of 920 tiles; the table has room for 4,256
    "grounds": lambda: grounds(20),  # clipped: fans of several sub-triangles
    "ground_behind_patch": lambda: join([patch(40, 3.0, -2.0), grounds(2)]),
    "walls_behind_patch": lambda: join([patch(40, 3.0, -2.0), walls(12)]),
    "everything": lambda: join([patch(9, 0.7, -2.0), walls(3), grounds(3, y=-0.6), patch(200, 3.0, -9.0, 3)]),
}


@pytest.mark.parametrize("W,H", [(640, 360), (333, 31)])
@pytest.mark.parametrize("name", sorted(SCENES))
def test_large_triangles(F, view, name, W, H):  # noqa: F811
    pos, idx = SCENES[name]()
    M = forward(W, H)
    v = view((pos, idx), M, W, H)
    for flags in (0, F.FA_VIS_CONSERVATIVE):
        want = O.visibility(M, pos, idx, W, H, conservative=bool(flags))
        assert want.any() and (v.bits(flags) == want).all()


@pytest.mark.parametrize("flags", [0, 2])
def test_more_fans_than_records(F, view, flags):  # noqa: F811
    """3,000 clipped triangles, of two large sub-triangles and more each: records for 4,024."""
    W, H = 96, 64
    pos, idx = grounds(1500, step=0.0005)
    M = forward(W, H)
    assert (view((pos, idx), M, W, H).bits(flags) == O.visibility(M, pos, idx, W, H, conservative=flags != 0)).all()


def test_more_large_triangles_than_records(F, view):  # noqa: F811
    """1.06M triangles of 17x17 pixel boxes and a thousand that fill the window: records for 2^20."""
    W, H, n = 1280, 720, 1060000
    rng = np.random.default_rng(7)
    at = rng.uniform((0.0, 0.0), (W - 18.0, H - 18.0), (n, 2))
    z = rng.uniform(-0.9, 0.9, n)
    px = np.stack([at, at + (16.9, 0.0), at + (0.0, 16.9)], 1)
    big = np.array([(-W, -H), (3 * W, -H), (-W, 3 * H)], np.float64)
    px[:: n // 1000] = big
    z[:: n // 1000] = np.linspace(0.5, 0.99, len(z[:: n // 1000]))
    pos = np.concatenate([px * (2.0 / W, 2.0 / H) - 1.0, np.repeat(z, 3).reshape(n, 3, 1)], 2)
    pos = pos.reshape(-1, 3).astype(np.float32)
    idx = np.arange(3 * n, dtype=np.uint32).reshape(-1, 3)
    M = np.eye(4, dtype=np.float32)
    want = O.visibility(M, pos, idx, W, H)
    assert want.any() and (view((pos, idx), M, W, H).bits() == want).all()


@pytest.mark.parametrize("name", ["walls", "grounds", "ground_behind_patch"])
def test_large_triangles_time(F, view, name):  # noqa: F811
    """Large triangles are shared by the whole grid: no slower than two rasterizations (half as fast again is
    left for the clock's steps)."""
    W, H = 960, 540
    v = view(SCENES[name](), forward(W, H), W, H)
    one, two = v.ms(), v.ms(raster=F.FA_RASTER_HIZ)
    assert one <= 1.5 * two + 0.02, (one, two)
