"""pc_timing: each pass has its own time, and the frames timed are the oracle's."""
import numpy as np
import pytest

import oracle as O
import paper_2204_01287_gb300 as pcr
import pcsynth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [4, 10240])
def test_the_clear_is_timed_by_itself(cuda_lib, batch):
    import torch
    p = S.terrain_params(1000.0, 0.2, 30)
    xyz, rgba = S.terrain(100_000, p, seed=2)
    W = H = 8192
    with pcr.Context(0, batch_size=batch) as ctx:
        cloud = ctx.upload(xyz, rgba)
        v = pcr.make_view(S.overview(p, W, H), W, H, pcr.PC_VIEW_CULL)
        fb = ctx.framebuffers([v])
        for _ in range(3):
            ctx.render(cloud, [v], fb)
        plain, st = fb[0][0].clone(), ctx.stats()
        torch.cuda.synchronize()
        pcr.pc_timing_begin(ctx.h)
        for _ in range(4):
            ctx.render(cloud, [v], fb)
        torch.cuda.synchronize()
        t = pcr.pc_timing_end(ctx.h)
        assert t.frames == 4
        assert torch.equal(fb[0][0], plain)
        # 8,192 x 8,192 keys of 8 bytes: what does not stay in 129 MB of L2 leaves at
        # 7.9 TB/s at most
        least = (8.0 * W * H - 129e6) / 7.9e12 * 1e3
        assert t.ms_clear / 4 > least
        # 25,000 batches at most are tested in much less than that
        assert t.ms_cull / 4 < least
        assert ctx.stats()["points_k"] == st["points_k"] and st["points_processed"] > 50_000


def test_a_view_of_an_empty_cloud_is_timed(cuda_lib):
    import torch
    with pcr.Context(0) as ctx:
        cloud = ctx.upload(np.zeros((0, 3), np.float32), np.zeros(0, np.uint32))
        v = pcr.make_view(S.cube_camera(64, 48), 64, 48)
        pcr.pc_timing_begin(ctx.h)
        [(vis, img)] = ctx.render(cloud, [v])
        torch.cuda.synchronize()
        t = pcr.pc_timing_end(ctx.h)
        assert t.frames == 1 and (pcr.vis_to_numpy(vis) == O.EMPTY).all()
        assert not pcr.rgba_to_numpy(img).any()
