"""Device memory of a context: the depth buffer of the single rasterization (8 bytes a pixel) shares its memory
with the chart and pack passes' scratch, so that a context of a usual window and chart count takes no more than
one with a 4-byte depth buffer of its own took.
"""
import pytest

from test_gpu_parity import F  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def own_buffers(T, V, C, W, H):
    """Bytes of a context whose parts are allocations of their own, the depth buffer 4 bytes a pixel: those of a
    megabyte and more take whole 2 MB steps."""
    up = lambda a, b: -(-a // b)  # noqa: E731
    blocks, front = up(T, 1024) + 1, T + 152 * 4 * 512
    queue = min(T + 1024, 1 << 20)
    chunks = up(C, 4096)
    raster = [4 * W * H, W * H // 64, queue * 64, queue * 16, (front + 65536) * 48, front * 4, front * 48, front * 4]
    charts = [4 * (T + V), T // 4, blocks * 4, blocks * 4, blocks * 24 * 1024, 8 * T, 16 * C, 4 * C]
    pack = [up(C, 1024) * 4 * 8192, 4 * C, 4 * C, chunks * 4096 * 8, 64 * chunks * 4096 * 8, 64 * chunks * 4104 * 2,
            64 * chunks * 8, 64 * 8 * C]
    return sum(up(n, 2 << 20) * (2 << 20) if n >= 1 << 20 else n for n in raster + charts + pack)


@pytest.mark.parametrize("T,C,W,H", [(7938, 1 << 14, 480, 270), (7938, 1 << 14, 2560, 1440), (100000, 1 << 15, 1920, 1080),
                                     (100000, 1 << 14, 3840, 2160), (100000, 1 << 15, 3840, 2160),
                                     (2000000, 1 << 16, 3840, 2160)])
def test_context_memory(F, T, C, W, H):  # noqa: F811
    import torch
    torch.zeros(1, device="cuda")
    make = lambda: F.Context(max_tris=T, max_verts=T // 2, max_charts=C, max_width=W, max_height=H)  # noqa: E731
    make().close()
    before = torch.cuda.mem_get_info()[0]
    ctxs = [make() for _ in range(3)]
    each = (before - torch.cuda.mem_get_info()[0]) / 3
    for c in ctxs:
        c.close()
    assert each <= own_buffers(T, T // 2, C, W, H)
