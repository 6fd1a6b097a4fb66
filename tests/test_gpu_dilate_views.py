"""The dilating resolve's grid holds the tiles of the views that dilate into an image,
and of no others: views of many sizes, plain ones and ones without an image beside
them, in any order."""
import numpy as np
import pytest

import oracle as O
import paper_2204_01287_gb300 as pcr
import pcsynth as S

pytestmark = pytest.mark.gpu

D, P, N = "dilated", "plain", "no image"


@pytest.mark.parametrize("kinds", [(D,), (N,), (N, N), (N, D), (D, N), (P, D), (D, P, N), (P, N), (N, P, D, D),
                                   (D,) * 9, (P, D) * 16, (N, D, P, D) * 8])
def test_views_beside_one_another(cuda_lib, kinds):
    import torch
    p = S.terrain_params(1000.0, 0.2, 30)
    xyz, rgba = S.terrain(30_000, p, seed=2)
    enc = O.encode(xyz, rgba, 1024)
    sizes = [(1 + (37 * i) % 150, 1 + (61 * i) % 100) for i in range(len(kinds))]
    sizes[len(kinds) // 2] = (257, 129)
    with pcr.Context(0, batch_size=1024) as ctx:
        cloud = ctx.upload(xyz, rgba)
        ms = [S.random_view(p, i, w, h, seed=2) for i, (w, h) in enumerate(sizes)]
        views = [pcr.make_view(m, w, h, pcr.PC_VIEW_CULL | (0 if k == P else pcr.PC_VIEW_DILATE))
                 for k, m, (w, h) in zip(kinds, ms, sizes)]
        fbs = ctx.framebuffers(views)
        bufs = [(v.data_ptr(), 0 if k == N else i.data_ptr()) for k, (v, i) in zip(kinds, fbs)]
        stream = torch.cuda.current_stream().cuda_stream
        torch.cuda.synchronize()
        for _ in range(2):   # the second frame's counters start from zero
            pcr.pc_render(ctx.h, cloud, views, bufs, stream)
        torch.cuda.synchronize()
        for i, (k, m, (w, h)) in enumerate(zip(kinds, ms, sizes)):
            ovis, st = O.render(enc, O.make_view(m, w, h, cull=True))
            assert np.array_equal(pcr.vis_to_numpy(fbs[i][0]), ovis), i
            assert ctx.stats(i)["points_k"] == st["points_k"]
            if k == D:
                ref = O.resolve_dilated(ovis, w, h, enc.color)
            elif k == P:
                ref = O.resolve(ovis, enc.color)
            else:
                continue
            assert np.array_equal(pcr.rgba_to_numpy(fbs[i][1]), ref), i
