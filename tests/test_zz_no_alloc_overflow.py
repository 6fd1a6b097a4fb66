"""pc_render_noalloc with more segments than its static draw list holds (batches that
overlap in the caller's buffers): the error word says so, and exactly what fits is
drawn, from either end of the list and from both."""
import numpy as np
import pytest

import oracle as O
import paper_2204_01287_gb300 as pcr
import pcsynth as S
from test_zz_no_alloc import _device_batches, _device_words, _render

pytestmark = pytest.mark.gpu

W, H = 64, 48
ENTRIES = 1 << 17


@pytest.mark.parametrize("kind", ["certified", "general", "both"])
def test_what_fits_is_drawn(cuda_lib, kind):
    import torch
    xyz, rgba = S.unit_cube(1 << 20, seed=2)
    enc = O.encode(xyz, rgba, 10240)
    words = [_device_words(torch, a) for a in (enc.w1, enc.w2, enc.w3, enc.color)]
    whole = enc.batches[:1].copy()   # 512 segments of 2,048 points
    whole["min"] = xyz.min(axis=0)
    whole["size"] = xyz.max(axis=0) - xyz.min(axis=0)
    whole["first"], whole["count"] = 0, enc.n
    # the whole cube lies inside the view, or has the eye inside it; 5 segments in a
    # small box far from the eye are inside the view either way
    m = S.cube_camera(W, H) if kind == "certified" else \
        S.look_at_perspective((0.5, 0.5, 0.9), (0.5, 0.5, 0.0), (0, 1, 0), 60.0, W / H, 0.01, 10.0)
    small = enc.batches[:1].copy()
    small["min"], small["size"] = (0.45, 0.45, 0.1), (0.1, 0.1, 0.1)
    parts = [(whole, 300)] if kind != "both" else [(whole, 150), (small, 12_000)]
    batches = np.concatenate([np.repeat(b, times) for b, times in parts])
    segments = sum(times * -(-int(b["count"][0]) // 2048) for b, times in parts)
    # some of every kind fit: what is too much is less than each kind's entries
    assert ENTRIES < segments and all(segments - ENTRIES < times * -(-int(b["count"][0]) // 2048)
                                      for b, times in parts)
    ref = O.Encoded(np.concatenate([b for b, _ in parts]), enc.w1, enc.w2, enc.w3, enc.color, enc.perm)
    ovis, _ = O.render(ref, O.make_view(m, W, H))
    err = np.zeros(2, np.uint32)
    vis, img = _render(pcr.lib(), torch, _device_batches(torch, batches), len(batches), words, enc.n,
                       pcr.make_view(m, W, H), err)
    assert err[0] == 1 and err[1] >= ENTRIES
    assert (ovis != O.EMPTY).sum() > 0.2 * W * H
    assert np.array_equal(vis, ovis)
    assert np.array_equal(img, O.resolve(ovis, enc.color))
    # the next good call is clean again
    vis, _ = _render(pcr.lib(), torch, _device_batches(torch, enc.batches), len(enc.batches), words,
                     enc.n, pcr.make_view(m, W, H), err)
    assert err[0] == 0 and np.array_equal(vis, O.render(enc, O.make_view(m, W, H))[0])
