"""The dilating resolve (Sec. 3.7) against the oracle, at the sizes where its
tiles of 32x32 pixels and their borders end, with equal depths everywhere (the
index then decides) and with sparse images (empty windows)."""
import numpy as np
import pytest

import oracle as O
import paper_2204_01287_gb300 as pcr
import pcsynth as S

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (31, 33), (32, 32), (33, 65), (70, 5), (3, 100), (129, 97)]


def _plane(n, seed, flat):
    """Points on the plane z = 0 (one depth for a camera along -z), or in a slab."""
    r = np.random.default_rng(seed)
    xyz = r.uniform(-1, 1, (n, 3)).astype(np.float32)
    if flat:
        xyz[:, 2] = 0.0
    return xyz, r.integers(0, 2**32, n, dtype=np.uint32)


@pytest.mark.parametrize("flat", [True, False])
@pytest.mark.parametrize("n", [60, 20_000])
@pytest.mark.parametrize("flag", [0, pcr.PC_VIEW_HQS, pcr.PC_VIEW_HQS_PACKED])
def test_dilated_tiles_match_oracle(cuda_lib, flag, n, flat):
    import torch
    xyz, rgba = _plane(n, 3, flat)
    enc = O.encode(xyz, rgba, 1024)
    with pcr.Context(0, batch_size=1024) as ctx:
        cloud = ctx.upload(xyz, rgba)
        # dilated views of every size, and one plain view, in one launch
        ms = [S.look_at_perspective((0, 0, 2), (0, 0, 0), (0, 1, 0), 60.0, W / H, 0.1, 10.0)
              for W, H in SIZES]
        views = [pcr.make_view(m, W, H, pcr.PC_VIEW_DILATE | flag) for m, (W, H) in zip(ms, SIZES)]
        views.append(pcr.make_view(ms[-1], 64, 48, flag))
        fbs = ctx.render(cloud, views)
        torch.cuda.synchronize()
        for m, (W, H), (vis, img) in zip(ms + [ms[-1]], SIZES + [(64, 48)], fbs):
            ov = O.make_view(m, W, H)
            ovis, _ = O.render(enc, ov)
            assert np.array_equal(pcr.vis_to_numpy(vis), ovis)
            shaded = O.render_hqs(enc, ov, ovis) if flag else None
            if (W, H) == (64, 48):
                ref = shaded if flag else O.resolve(ovis, enc.color)
            elif flag:
                ref = O.hqs_resolve_dilated(ovis, W, H, shaded)
            else:
                ref = O.resolve_dilated(ovis, W, H, enc.color)
            assert np.array_equal(pcr.rgba_to_numpy(img), ref), (W, H)
