"""Small images of long draw lists take their entries another way than larger ones and
short lists: both sides of the line (16,384 pixels; as many entries as warps) against
the oracle, with certified and other batches."""
import numpy as np
import pytest

import oracle as O
import paper_2204_01287_gb300 as pcr
import pcsynth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=[30_000, 400_000])
def world(request):
    """Batches of 32 points: 938 entries, a short list, or 12,500, a long one."""
    p = S.terrain_params(3000.0, 0.2, 60)
    xyz, rgba = S.terrain(request.param, p, seed=9)
    return p, xyz, rgba, O.encode(xyz, rgba, 32)


@pytest.mark.parametrize("shape", [{}, {"threads_per_block": 32, "blocks_per_sm": 1}])
@pytest.mark.parametrize("size", [(1, 1), (16, 9), (128, 128), (127, 129), (128, 129)])
def test_both_ways_match_oracle(cuda_lib, world, size, shape):
    import torch
    p, xyz, rgba, enc = world
    W, H = size
    h = S.terrain_height(p, 0.0, 0.0)
    # certified batches, both kinds, and (without the early-depth test) none certified
    views = [(S.overview(p, W, H), 0), (S.flythrough(p, 10, 120, W, H, seed=9), 0),
             (S.look_at_perspective((0, 0, h + 2), (100, 30, h), (0, 0, 1), 70.0, W / H, 0.5, 1e5), 0),
             (S.overview(p, W, H), pcr.PC_VIEW_NO_EARLY_DEPTH)]
    with pcr.Context(0, batch_size=32, **shape) as ctx:
        cloud = ctx.upload(xyz, rgba)
        for m, flags in views:
            for _ in range(2):
                [(vis, img)] = ctx.render(cloud, [pcr.make_view(m, W, H, pcr.PC_VIEW_CULL | flags)])
            torch.cuda.synchronize()
            ovis, st = O.render(enc, O.make_view(m, W, H, cull=True))
            assert np.array_equal(pcr.vis_to_numpy(vis), ovis)
            assert np.array_equal(pcr.rgba_to_numpy(img), O.resolve(ovis, enc.color))
            assert ctx.stats()["points_k"] == st["points_k"]
