"""The schedule autotuners try each raster schedule once: the mid-size limit is part of the tile-depth option's
second rasterization, so without that option there is one schedule."""
import pytest

from paper_2502_17712_gb300 import scenes as S
from test_gpu_parity import F  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def test_tuners_try_each_raster_schedule_once(F):  # noqa: F811
    sc = S.grid_scene(1, 33)
    batch = F.Batch(1, max_tris=sc.T, max_verts=sc.V, max_charts=1 << 12, max_width=320, max_height=200,
                    max_atlas_log2=10)
    mesh = F.BatchMesh(batch, sc.pos, sc.idx)
    params = [F.frame_params(S.hemisphere_camera(1, 320, 200), 320, 200, 1.0, 10)]
    bufs = [F.FrameBuffers.allocate(sc.T, sc.V, 1 << 12)]
    plan = F.BatchPlan(batch, [mesh], params, bufs)
    before = batch.launches
    plan.tune(reps=1)
    # a warm-up and a timed launch of 3 raster schedules and, on one lane, 3 worker counts
    assert batch.launches - before == 2 * (3 + 3)
    for _ in range(6):
        lanes, policy, pct, mid, flags, ms = plan.tune(reps=1)
        assert mid == F.FA_RASTER_MID_OFF or flags == F.FA_RASTER_HIZ
        F.batch_tune(batch, [mesh], params, bufs, reps=1)
        k = batch.kernel_schedule()
        assert k["mid_max_pix"] == F.FA_RASTER_MID_OFF or k["raster_flags"] == F.FA_RASTER_HIZ
    plan.close()
    mesh.close()
    batch.close()
