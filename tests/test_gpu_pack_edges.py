"""The packer at the box counts where its work is divided differently: one order tile
(1,024 boxes), one chunk (4,096, scanned by the candidates' own CTAs), and the counts
beside them, for every push shape, against the oracle (integers, compared exactly).
"""
import numpy as np
import pytest

import oracle as O
from paper_2502_17712_gb300 import scenes as S
from test_gpu_parity import F  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("push", [256, 512, 1024])
@pytest.mark.parametrize("n", [1, 33, 1023, 1024, 1025, 4095, 4096, 4097])
def test_pack_counts(F, n, push):  # noqa: F811
    import torch
    log2 = 11
    ctx = F.Context(max_tris=64, max_verts=64, max_charts=8192, max_width=64, max_height=64)
    ctx.set_chart_pack_schedule(push_threads=push)
    for seed, scales in ((n, 64), (n + 1, 8)):
        fa, fb = S.lognormal_boxes(seed, n, mean_texels=8)
        if n > 40:  # many boxes of one height: the order inside a bin is the boxes' own
            fb[: n // 2] = np.maximum(fa[: n // 2], 2560)
        d_fa, d_fb = (torch.as_tensor(x.view(np.int32)).cuda() for x in (fa, fb))
        cnt = torch.tensor([n], dtype=torch.int32, device="cuda")
        order = torch.zeros(n, dtype=torch.int32, device="cuda")
        place = torch.zeros(n, 4, dtype=torch.int32, device="cuda")
        res = torch.zeros(5, dtype=torch.int32, device="cuda")
        F.fa_pack(ctx.handle, d_fa, d_fb, cnt, log2, scales, 0, order, place, res)
        torch.cuda.synchronize()
        pk = O.pack(fa, fb, log2, n_scales=scales)
        r = res.cpu().numpy().view(np.uint32)
        assert pk.status == 0 and (int(r[3]), int(r[4])) == (0, n)
        assert (int(r[0]), int(r[1]), int(r[2])) == (pk.k, pk.omega, pk.height)
        assert (place.cpu().numpy() == pk.place).all()
        assert (order.cpu().numpy() == O.order(fb)).all()
    ctx.close()
