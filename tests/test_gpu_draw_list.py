"""One-view launches split the draw list: certified batches (the list's front)
and the others (its back) are drawn by two kernels that may overlap. Frames
that mix both, at the sizes where segments, steps and groups end, must be
bit-identical to the oracle, also back to back on one stream and as replayed
graphs."""
import numpy as np
import pytest

import oracle as O
import paper_2204_01287_gb300 as pcr
import pcsynth as S

pytestmark = pytest.mark.gpu

W, H = 333, 201


def _views(p):
    """Everything inside the view, batches across its edges, and the eye
    among the points (batches on both sides of the eye plane)."""
    h = S.terrain_height(p, 0.0, 0.0)
    return [S.overview(p, W, H), S.random_view(p, 3, W, H, seed=4),
            S.look_at_perspective((0, 0, h + 2), (100, 30, h), (0, 0, 1), 70.0, W / H, 0.5, 1e5)]


@pytest.mark.parametrize("graphs", [False, True])
@pytest.mark.parametrize("n,batch", [(1, 128), (127, 128), (129, 128), (4097, 1024),
                                     (40_961, 1028), (300_003, 10240)])
def test_mixed_lists_match_oracle(cuda_lib, n, batch, graphs):
    import torch
    p = S.terrain_params(3000.0, 0.2, 60)
    xyz, rgba = S.terrain(n, p, seed=4)
    enc = O.encode(xyz, rgba, batch)
    stream = torch.cuda.Stream()
    with pcr.Context(0, batch_size=batch, flags=pcr.PC_CFG_GRAPHS if graphs else 0) as ctx:
        cloud = ctx.upload(xyz, rgba)
        views = [pcr.make_view(m, W, H, pcr.PC_VIEW_CULL) for m in _views(p)]
        fbs = [ctx.framebuffers([v]) for v in views]
        for _ in range(3):   # nothing waits between the frames
            for v, fb in zip(views, fbs):
                ctx.render(cloud, [v], fb, stream=stream)
        torch.cuda.synchronize()
        for v, [(vis, img)] in zip(views, fbs):
            ovis, st = O.render(enc, O.make_view(np.array(v.view_proj), W, H, cull=True))
            assert np.array_equal(pcr.vis_to_numpy(vis), ovis)
            assert np.array_equal(pcr.rgba_to_numpy(img), O.resolve(ovis, enc.color))
            ctx.render(cloud, [v], fbs[0], stream=stream)
            gst = ctx.stats(stream=stream)
            assert gst["batches_k"] == st["batches_k"]
            assert gst["points_atomic"] >= (ovis != O.EMPTY).sum()
