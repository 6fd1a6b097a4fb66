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


@pytest.mark.parametrize("nviews", [1, 2, 3, 5, 31, 32])
@pytest.mark.parametrize("n,batch", [(3, 4), (31 * 8 + 5, 8), (33 * 8, 8), (1029, 8), (130_001, 64)])
def test_cull_blocks_match_oracle(cuda_lib, n, batch, nviews):
    """Counts of batches and views around the cull pass's blocks and rounds:
    every view's image and counters are the oracle's."""
    import torch
    p = S.terrain_params(2000.0, 0.2, 30)
    xyz, rgba = S.terrain(n, p, seed=6)
    enc = O.encode(xyz, rgba, batch)
    with pcr.Context(0, batch_size=batch) as ctx:
        cloud = ctx.upload(xyz, rgba)
        ms = [S.random_view(p, i, 40 + i, 33, seed=6) if i % 3 else S.overview(p, 40 + i, 33)
              for i in range(nviews)]
        views = [pcr.make_view(m, 40 + i, 33, pcr.PC_VIEW_CULL) for i, m in enumerate(ms)]
        fbs = ctx.render(cloud, views)
        torch.cuda.synchronize()
        for i in range(0, nviews, 5):
            ovis, st = O.render(enc, O.make_view(ms[i], 40 + i, 33, cull=True))
            assert np.array_equal(pcr.vis_to_numpy(fbs[i][0]), ovis)
            gst = ctx.stats(i)
            assert gst["batches_k"] == st["batches_k"]
            assert gst["points_k"] == st["points_k"]


def test_statistics_survive_a_separate_resolve(cuda_lib):
    """pc_resolve draws nothing, so the last frame's counters stay; the next
    frame's start from zero."""
    import torch
    p = S.terrain_params(2000.0)
    xyz, rgba = S.terrain(50_000, p, seed=7)
    with pcr.Context(0) as ctx:
        cloud = ctx.upload(xyz, rgba)
        v = pcr.make_view(S.overview(p, 80, 50), 80, 50, pcr.PC_VIEW_CULL)
        fbs = ctx.render(cloud, [v])
        st = ctx.stats()
        ctx.resolve(cloud, [v], fbs)
        assert ctx.stats() == st and st["points_processed"] == 50_000
        ctx.render(cloud, [v], fbs)
        torch.cuda.synchronize()
        assert ctx.stats()["points_k"] == st["points_k"]


@pytest.mark.parametrize("nviews", [2, 3, 5, 8, 17])
@pytest.mark.parametrize("n,batch", [(300, 8), (300_000, 10240)])
def test_views_with_and_without_culling_share_a_warp(cuda_lib, n, batch, nviews):
    """Views of one launch that differ in culling and forced precision: the
    teams of a warp test batches for views of both kinds."""
    import torch
    p = S.terrain_params(4000.0, 0.2, 60)
    xyz, rgba = S.terrain(n, p, seed=1)
    enc = O.encode(xyz, rgba, batch)
    W, H = 160, 90
    with pcr.Context(0, batch_size=batch) as ctx:
        cloud = ctx.upload(xyz, rgba)
        ms = [S.flythrough(p, 10 * i, 120, W, H, seed=1) if i % 3 else S.cube_camera(W, H)
              for i in range(nviews)]
        ks = [i % 4 for i in range(nviews)]
        views = [pcr.make_view(m, W, H, (pcr.PC_VIEW_CULL if i % 2 else 0) | pcr.PC_VIEW_FORCE_K(k))
                 for i, (m, k) in enumerate(zip(ms, ks))]
        fbs = ctx.render(cloud, views)
        torch.cuda.synchronize()
        for i, (m, k) in enumerate(zip(ms, ks)):
            ovis, st = O.render(enc, O.make_view(m, W, H, cull=bool(i % 2), force_k=k))
            assert np.array_equal(pcr.vis_to_numpy(fbs[i][0]), ovis), i
            assert ctx.stats(i)["batches_k"] == st["batches_k"]
