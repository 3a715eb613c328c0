"""Mid-size boxes of the second rasterization (fa_set_raster_schedule's mid_max_pix with FA_RASTER_HIZ, the only
schedule that reads it): in-thread or in tiles, the frame is the oracle's, bit for bit."""
import numpy as np
import pytest

from paper_2502_17712_gb300 import scenes as S
from test_gpu_parity import F, compare_frame, run_gpu, small_ctx  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mid", [64, 256])
def test_mid_size_boxes(F, small_ctx, mid):  # noqa: F811
    """More survivors than the lane groups take: a thread each, a warp's mid-size boxes in-thread where cheaper."""
    sc = S.instanced_grid_scene(13, 24, n=32, half=3.0)
    M = S.hemisphere_camera(13, 1920, 1080, radius=4.0)
    mesh = F.Mesh(small_ctx, sc.pos, sc.idx)
    for flags in (0, F.FA_VIS_CONSERVATIVE):
        small_ctx.set_raster_schedule(mid, F.FA_RASTER_HIZ)
        try:
            b, st = run_gpu(F, small_ctx, mesh, M, 1920, 1080, 1.0, 11, flags=flags)
        finally:
            small_ctx.set_raster_schedule()
        assert small_ctx.frame_stats()["survivors"] > 9728
        compare_frame(sc, M, 1920, 1080, 1.0, 11, b, st, flags=flags)
    mesh.close()


@pytest.mark.parametrize("seed", range(4))
def test_mid_size_boxes_grouped(F, small_ctx, seed):  # noqa: F811
    """Few survivors: a lane group each."""
    rng = np.random.default_rng([seed, 0x6A1])
    sc = S.instanced_grid_scene(300 + seed, int(rng.integers(1, 5)), n=int(rng.choice([16, 24, 32])), half=2.0)
    W, H = [(640, 360), (1280, 720), (1920, 1080), (480, 270)][seed]
    M = S.hemisphere_camera(400 + seed, W, H, radius=float(rng.uniform(1.5, 4.0)))
    mesh = F.Mesh(small_ctx, sc.pos, sc.idx)
    small_ctx.set_raster_schedule(64, F.FA_RASTER_HIZ)
    try:
        b, st = run_gpu(F, small_ctx, mesh, M, W, H, 1.0, 11, flags=F.FA_VIS_CONSERVATIVE if seed % 2 else 0)
    finally:
        small_ctx.set_raster_schedule()
    compare_frame(sc, M, W, H, 1.0, 11, b, st, flags=F.FA_VIS_CONSERVATIVE if seed % 2 else 0)
    mesh.close()
