"""The first pass tests few batches with a team of lanes each and many (from 16,384)
with one thread each: both sides of that line against the oracle, for every kind of
view, for boxes on the clip planes and for the nodes of an LOD tree."""
import numpy as np
import pytest

import oracle as O
import paper_2204_01287_gb300 as pcr
import pcsynth as S
from test_gpu_cull import _boxes_on_planes

pytestmark = pytest.mark.gpu

LINE = 16384
W, H = 80, 60


def _views(p, n):
    """Views with and without culling, adaptive and forced precision, near and far."""
    out = []
    for i in range(n):
        m = S.overview(p, W, H) if i % 3 == 1 else S.random_view(p, i, W, H, seed=6) if i % 3 else \
            S.flythrough(p, 10 * i, 120, W, H, seed=6)
        out.append((m, i % 4 != 3, 0 if i % 5 else (i // 5 + 1) % 4))
    return out


@pytest.mark.parametrize("nviews", [1, 2, 5, 32])
@pytest.mark.parametrize("batches", [LINE - 1, LINE, LINE + 1, LINE + 127, 2 * LINE + 33])
def test_frames_on_both_sides_of_the_line(cuda_lib, batches, nviews):
    import torch
    p = S.terrain_params(2000.0, 0.2, 30)
    xyz, rgba = S.terrain(4 * batches - 1, p, seed=6)   # the last batch is ragged
    enc = O.encode(xyz, rgba, 4)
    assert len(enc.batches) == batches
    with pcr.Context(0, batch_size=4) as ctx:
        cloud = ctx.upload(xyz, rgba)
        vs = _views(p, nviews)
        fbs = ctx.render(cloud, [pcr.make_view(m, W, H, (pcr.PC_VIEW_CULL if cull else 0) | pcr.PC_VIEW_FORCE_K(k))
                                 for m, cull, k in vs])
        torch.cuda.synchronize()
        for i in sorted({0, 1, 3, 4, nviews // 2, nviews - 1} & set(range(nviews))):
            m, cull, k = vs[i]
            ovis, st = O.render(enc, O.make_view(m, W, H, cull=cull, force_k=k))
            assert np.array_equal(pcr.vis_to_numpy(fbs[i][0]), ovis), i
            got = ctx.stats(i)
            assert got["batches_k"] == st["batches_k"] and got["points_k"] == st["points_k"], i


@pytest.mark.parametrize("rel", [0.0, 1e-8, 1e-6, 1e-4])
@pytest.mark.parametrize("batches", [LINE - 384, LINE + 3616])
def test_culling_decisions_near_planes(cuda_lib, batches, rel):
    import torch
    rng = np.random.default_rng(int(rel * 1e9) + 5)
    ms = [S.cube_camera(64, 48), S.look_at_perspective((3, -2, 1), (0, 0.5, 0.2), (0, 0, 1), 40.0, 1.5, 0.5, 50.0)]
    with pcr.Context(0) as ctx:
        b = np.concatenate([_boxes_on_planes(m, batches // 2, rng, rel) for m in ms])
        b["first"] = np.arange(len(b), dtype=np.uint32) * 4
        n = 4 * len(b)
        words = rng.integers(0, 1 << 30, n, dtype=np.uint32)
        cloud = ctx.upload_encoded(b, words, words, words, np.zeros(n, np.uint32))
        ctx.render(cloud, [pcr.make_view(m, 64, 48, pcr.PC_VIEW_CULL) for m in ms])
        torch.cuda.synchronize()
        for i, m in enumerate(ms):
            ov = O.make_view(m, 64, 48, cull=True)
            expect = sum(not O.cull(bt, ov) for bt in b)
            assert 0 < expect < len(b)
            assert ctx.stats(i)["batches_rendered"] == expect


def test_nodes_of_a_large_tree(cuda_lib):
    import torch
    p = S.terrain_params(3000.0, 0.2, 60)
    xyz, rgba = S.terrain(300_000, p, seed=3)
    enc = O.encode(xyz, rgba, 10240)
    with pcr.Context(0) as ctx:
        lod = pcr.pc_build_lod(ctx.h, ctx.upload(xyz, rgba), 14, 8, 7)
        ref = O.lod_build(O.decode_cloud(enc, 3), enc.color, 14, 8, 7)
        assert len(ref.nodes) > LINE
        vs = [(S.flythrough(p, 20 * i, 120, W, H, seed=3), (0.0, 1.0, 4.0)[i % 3], (0.0, 12.0)[i % 2]) for i in range(6)]
        for group in (vs[:1], vs):
            fbs = ctx.render(lod, [pcr.make_view(m, W, H, pcr.PC_VIEW_CULL, px, far) for m, px, far in group])
            torch.cuda.synchronize()
            for i, (m, px, far) in enumerate(group):
                ovis, st = O.lod_render(ref, O.make_view(m, W, H), px, far)
                assert np.array_equal(pcr.vis_to_numpy(fbs[i][0]), ovis), i
                got = ctx.stats(i)
                assert got["batches_rendered"] == st["batches_rendered"] and got["batches_k"] == st["batches_k"], i
