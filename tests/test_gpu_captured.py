"""Frames that a caller captures into a CUDA graph (in every capture mode) and replays,
with eager frames of other lists between the replays: each image is the oracle's, and
the counters are each frame's own."""
import numpy as np
import pytest

import oracle as O
import paper_2204_01287_gb300 as pcr
import pcsynth as S

pytestmark = pytest.mark.gpu

W, H = 200, 150


@pytest.fixture(scope="module")
def world():
    p = S.terrain_params(3000.0, 0.2, 60)
    xyz, rgba = S.terrain(300_000, p, seed=4)
    return p, xyz, rgba, O.encode(xyz, rgba, 512)


@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
@pytest.mark.parametrize("flags", [0, pcr.PC_VIEW_HQS, pcr.PC_VIEW_HQS_PACKED, pcr.PC_VIEW_NO_EARLY_DEPTH])
def test_replays_between_eager_frames(cuda_lib, world, flags, mode):
    import torch
    p, xyz, rgba, enc = world
    h = S.terrain_height(p, 0.0, 0.0)
    near = S.look_at_perspective((0, 0, h + 2), (100, 30, h), (0, 0, 1), 70.0, W / H, 0.5, 1e5)
    ms = [near, S.overview(p, W, H), S.flythrough(p, 10, 120, W, H, seed=4)]
    refs = []
    for m in ms:
        ov = O.make_view(m, W, H, cull=True)
        vis, st = O.render(enc, ov)
        shaded = flags & (pcr.PC_VIEW_HQS | pcr.PC_VIEW_HQS_PACKED)
        refs.append((vis, O.render_hqs(enc, ov, vis) if shaded else O.resolve(vis, enc.color), st))
    stream = torch.cuda.Stream()
    with pcr.Context(0, batch_size=512) as ctx:
        cloud = ctx.upload(xyz, rgba)
        views = [[pcr.make_view(m, W, H, pcr.PC_VIEW_CULL | flags)] for m in ms]
        fbs = [ctx.framebuffers(v) for v in views]
        torch.cuda.synchronize()
        for v, fb in zip(views, fbs):   # the scratch is there before the captures
            ctx.render(cloud, v, fb, stream=stream)
        torch.cuda.synchronize()
        graphs = []
        for v, fb in zip(views[:2], fbs):
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream, capture_error_mode=mode):
                ctx.render(cloud, v, fb, stream=stream)
            graphs.append(g)

        def check(i):
            torch.cuda.synchronize()
            assert np.array_equal(pcr.vis_to_numpy(fbs[i][0][0]), refs[i][0])
            assert np.array_equal(pcr.rgba_to_numpy(fbs[i][0][1]), refs[i][1])
            assert ctx.stats(stream=stream)["points_k"] == refs[i][2]["points_k"]

        for _ in range(4):
            for i in (0, 1, 2, 1, 1, 0):
                for vis, img in fbs[i]:
                    vis.zero_()
                    img.zero_()
                torch.cuda.synchronize()
                with torch.cuda.stream(stream):
                    if i < 2:
                        graphs[i].replay()
                    else:
                        ctx.render(cloud, views[2], fbs[2], stream=stream)
                check(i)
        with torch.cuda.stream(stream):   # nothing waits between them
            for i in (0, 1, 0, 2, 0, 1):
                if i < 2:
                    graphs[i].replay()
                else:
                    ctx.render(cloud, views[2], fbs[2], stream=stream)
        check(1)
