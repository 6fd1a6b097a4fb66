"""Frames back to back on one stream: each frame's fast kernel starts beside the
general one and must see its own draw list and its own cleared keys, not those of
the frame before (whose depths may be smaller and whose list may be longer)."""
import threading

import numpy as np
import pytest

import oracle as O
import paper_2204_01287_gb300 as pcr
import pcsynth as S

pytestmark = pytest.mark.gpu

W, H = 320, 200


def _world(n, seed):
    """A cloud, views of near and far things in turn, and their images."""
    p = S.terrain_params(3000.0, 0.2, 60)
    xyz, rgba = S.terrain(n, p, seed=seed)
    enc = O.encode(xyz, rgba, 1024)
    h = S.terrain_height(p, 0.0, 0.0)
    ms = [S.look_at_perspective((0, 0, h + 30), (10, 3, h), (0, 0, 1), 70.0, W / H, 0.5, 1e5),
          S.overview(p, W, H), S.random_view(p, 3, W, H, seed=seed), S.overview(p, W, H)]
    images = []
    for m in ms:
        vis, _ = O.render(enc, O.make_view(m, W, H, cull=True))
        images.append(O.resolve(vis, enc.color))
    return xyz, rgba, [pcr.make_view(m, W, H, pcr.PC_VIEW_CULL) for m in ms], images


def _frames(ctx, cloud, views, stream, rounds):
    """Frames into one visibility buffer, an image for each."""
    import torch
    vis = ctx.framebuffers(views[:1])[0][0]
    out = [[(vis, torch.empty(W * H, dtype=torch.int32, device="cuda"))] for _ in range(rounds * len(views))]
    torch.cuda.synchronize()
    for i, fb in enumerate(out):
        ctx.render(cloud, [views[i % len(views)]], fb, stream=stream)
    return [fb[0][1] for fb in out]


@pytest.mark.parametrize("n", [4_000, 400_000])
def test_alternating_frames_share_a_visibility_buffer(cuda_lib, n):
    import torch
    xyz, rgba, views, images = _world(n, 5)
    stream = torch.cuda.Stream()
    with pcr.Context(0, batch_size=1024) as ctx:
        got = _frames(ctx, ctx.upload(xyz, rgba), views, stream, 16)
        torch.cuda.synchronize()
        for i, img in enumerate(got):
            assert np.array_equal(pcr.rgba_to_numpy(img), images[i % len(views)]), i


def test_two_contexts_draw_on_one_stream(cuda_lib):
    """Two threads queue frames of contexts of their own on the same stream, so that
    one's kernels come between the other's."""
    import torch
    worlds = [_world(200_000, 7), _world(30_000, 8)]
    stream = torch.cuda.Stream()
    got = [None, None]
    ctxs = [pcr.Context(0, batch_size=1024) for _ in worlds]
    clouds = [c.upload(w[0], w[1]) for c, w in zip(ctxs, worlds)]

    def work(t):
        got[t] = _frames(ctxs[t], clouds[t], worlds[t][2], stream, 16)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for t, w in enumerate(worlds):
        for i, img in enumerate(got[t]):
            assert np.array_equal(pcr.rgba_to_numpy(img), w[3][i % 4]), (t, i)
    for c in ctxs:
        c.close()
