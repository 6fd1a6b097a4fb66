"""pc_render_noalloc captured into a caller's graph: replays, with other calls between
them, draw the oracle's frame (one branch, no frame number: the calls before and after
share the static scratch)."""
import ctypes

import numpy as np
import pytest

import oracle as O
import paper_2204_01287_gb300 as pcr
import pcsynth as S
from test_zz_no_alloc import _device_batches, _device_words, _render

pytestmark = pytest.mark.gpu

W, H = 160, 120


def test_replays_between_calls(cuda_lib):
    import torch
    p = S.terrain_params(3000.0, 0.2, 60)
    xyz, rgba = S.terrain(200_000, p, seed=4)
    enc = O.encode(xyz, rgba, 512)
    L = pcr.lib()
    words = [_device_words(torch, a) for a in (enc.w1, enc.w2, enc.w3, enc.color)]
    batches = _device_batches(torch, enc.batches)
    h = S.terrain_height(p, 0.0, 0.0)
    ms = [S.look_at_perspective((0, 0, h + 2), (100, 30, h), (0, 0, 1), 70.0, W / H, 0.5, 1e5),
          S.overview(p, W, H), S.flythrough(p, 10, 120, W, H, seed=4)]
    views = [pcr.make_view(m, W, H, pcr.PC_VIEW_CULL) for m in ms]
    refs = [O.render(enc, O.make_view(m, W, H, cull=True))[0] for m in ms]
    err = np.zeros(2, np.uint32)
    vis, _ = _render(L, torch, batches, len(enc.batches), words, enc.n, views[2], err)   # before any capture
    assert np.array_equal(vis, refs[2])
    bufs, graphs = [], []
    stream = torch.cuda.Stream()
    for v in views[:2]:
        a = torch.zeros(W * H, dtype=torch.int64, device="cuda")
        b = torch.zeros(W * H, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            assert L.pc_render_noalloc(batches.data_ptr(), len(enc.batches), *(w.data_ptr() for w in words), enc.n,
                                       ctypes.byref(v), a.data_ptr(), b.data_ptr(), 512.0, None,
                                       stream.cuda_stream) == pcr.PC_OK
        bufs.append((a, b))
        graphs.append(g)
    for _ in range(4):
        for i in (0, 1, 1, 2, 0):
            if i == 2:
                vis, img = _render(L, torch, batches, len(enc.batches), words, enc.n, views[2], err)
                assert err[0] == 0
            else:
                for t in bufs[i]:
                    t.zero_()
                torch.cuda.synchronize()
                graphs[i].replay()
                torch.cuda.synchronize()
                vis, img = pcr.vis_to_numpy(bufs[i][0]), pcr.rgba_to_numpy(bufs[i][1])
            assert np.array_equal(vis, refs[i])
            assert np.array_equal(img, O.resolve(refs[i], enc.color))
