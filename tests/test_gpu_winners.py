"""Single-pass visibility (the triangle of every pixel kept with its depth key)
against the oracle and against the second rasterization, which the tile-depth
option keeps: the same visible bits, also where many triangles tie at a pixel.
All outputs are bits, compared exactly.
"""
import numpy as np
import pytest

import oracle as O
from paper_2502_17712_gb300 import scenes as S
from test_gpu_parity import F  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def visible(F, pos, idx, M, W, H, flags=0):  # noqa: F811
    import torch
    ctx = F.Context(max_tris=idx.shape[0], max_verts=pos.shape[0], max_charts=16, max_width=W, max_height=H)
    ctx.set_raster_schedule(16, flags)
    mesh = F.Mesh(ctx, pos, idx)
    vt = torch.zeros((idx.shape[0] + 31) // 32, dtype=torch.int32, device="cuda")
    F.fa_visibility(ctx.handle, mesh.handle, M, W, H, vt)
    torch.cuda.synchronize()
    assert ctx.device_status() == F.FA_OK
    out = vt.cpu().numpy().view(np.uint32)
    mesh.close()
    ctx.close()
    return out


@pytest.mark.parametrize("copies", [1, 2, 5])  # 5: more ties than the list holds (131,072)
@pytest.mark.parametrize("n,radius", [(200, 1.6), (40, 1.6), (2, 1.6), (2, 0.3)])  # small, mid-size, large, clipped
def test_coplanar_stacks(F, copies, n, radius):  # noqa: F811
    """Copies of one patch at the same place: every copy of a visible triangle is visible."""
    sc = S.grid_scene(5, n)
    pos = np.concatenate([sc.pos] * copies)
    idx = np.concatenate([sc.idx + np.uint32(c * sc.V) for c in range(copies)])
    W = H = 400
    M = S.view_proj((0.1, -0.2, radius), (0.0, 0.0, 0.0), (0.0, 1.0, 0.0), W, H)
    vt = visible(F, pos, idx, M, W, H)
    want, z = O.visibility(M, pos, idx, W, H, return_zbuf=True)
    covered = int((z != 0xFFFFFFFF).sum())
    assert copies < 5 or (copies - 1) * covered > 131072
    assert want.any() and (vt == want).all()


@pytest.mark.parametrize("W,H", [(1, 1), (63, 33), (64, 32), (65, 31), (257, 129)])
def test_odd_windows(F, W, H):  # noqa: F811
    sc = S.instanced_grid_scene(3, 3, 33)
    M = S.hemisphere_camera(4, W, H, radius=5.0)
    vt = visible(F, sc.pos, sc.idx, M, W, H)
    assert (vt == O.visibility(M, sc.pos, sc.idx, W, H)).all()


@pytest.mark.parametrize("parts,n,W,H,radius", [(40, 64, 1920, 1080, 10.0), (300, 33, 2560, 1440, 7.0),
                                                (12, 17, 2559, 1439, 4.0), (100, 9, 1280, 720, 1.0)])
def test_equals_second_rasterization(F, parts, n, W, H, radius):  # noqa: F811
    """Overlapping floors: every box size, triangles past the window and the near plane, ties by chance."""
    sc = S.instanced_grid_scene(parts, parts, n)
    M = S.hemisphere_camera(parts, W, H, radius=radius)
    a, b = visible(F, sc.pos, sc.idx, M, W, H), visible(F, sc.pos, sc.idx, M, W, H, F.FA_RASTER_HIZ)
    assert a.any() and (a == b).all()


@pytest.mark.parametrize("parts,n,W,H,radius", [(1, 64, 480, 270, 3.0), (40, 33, 901, 613, 7.0), (8, 5, 640, 360, 3.0),
                                                (30, 9, 333, 222, 0.8), (2, 150, 63, 31, 6.0)])
def test_conservative_marking(F, parts, n, W, H, radius):  # noqa: F811
    """Conservative marking of what the samples left: small boxes, the warp's, clipped ones, triangles without a
    pixel centre; against the oracle, and against the second rasterization."""
    import torch
    sc = S.instanced_grid_scene(parts, parts, n, half=1.5)
    M = S.hemisphere_camera(parts + 5, W, H, radius=radius)
    want = O.visibility(M, sc.pos, sc.idx, W, H, conservative=True)
    ctx = F.Context(max_tris=sc.T, max_verts=sc.V, max_charts=16, max_width=W, max_height=H)
    mesh = F.Mesh(ctx, sc.pos, sc.idx)
    vt = torch.zeros((sc.T + 31) // 32, dtype=torch.int32, device="cuda")
    for flags in (0, F.FA_RASTER_HIZ):
        ctx.set_raster_schedule(16, flags)
        F.fa_visibility(ctx.handle, mesh.handle, M, W, H, vt, flags=F.FA_VIS_CONSERVATIVE)
        torch.cuda.synchronize()
        assert ctx.device_status() == F.FA_OK
        assert want.any() and (vt.cpu().numpy().view(np.uint32) == want).all()
    mesh.close()
    ctx.close()
