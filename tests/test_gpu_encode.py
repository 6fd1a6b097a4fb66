"""pc_upload_cloud encodes on the device; its cloud must be the host encoder's bit
for bit (boxes, words, colours), which tests elsewhere hold to the oracle. Sizes
around the sort's tiles and warps, every shape of tie, and the corner cases of
the binary32 box (signed zeros, one value, an overflowing size)."""
import numpy as np
import pytest

import paper_2204_01287_gb300 as pcr
import pcsynth as S

pytestmark = pytest.mark.gpu


def _cloud(kind, n):
    r = np.random.default_rng(n + 17)
    if kind == "terrain":
        return S.terrain(n, S.terrain_params(3000.0, 0.2, 40), seed=9)
    xyz = r.uniform(-5, 5, (n, 3)).astype(np.float32)
    if kind == "ties":          # few distinct positions: the sort must be stable
        xyz = np.floor(xyz).astype(np.float32)
    if kind == "flat":          # an axis without extent, another of zeros of both signs
        xyz[:, 1] = 2.5
        xyz[:, 2] = np.where(r.random(n) < 0.5, np.float32(0.0), np.float32(-0.0))
    if kind == "zeros":         # minima and maxima that are zeros of both signs
        xyz = np.abs(np.floor(xyz)).astype(np.float32) * np.float32([1, -1, 1])
        xyz = np.where((xyz == 0) & (r.random((n, 3)) < 0.5), np.float32(-0.0), xyz).astype(np.float32)
    if kind == "wide":          # the box's size overflows binary32
        xyz = (xyz * np.float32(6e37)).astype(np.float32)
    if kind == "tiny":          # subnormal coordinates
        xyz = (xyz * np.float32(1e-40)).astype(np.float32)
    return xyz, r.integers(0, 2**32, n, dtype=np.uint32)


def _same(ctx, cloud, host):
    got = pcr.pc_cloud_download(ctx.h, cloud)
    assert got[0].tobytes() == host[0].tobytes()
    for a, b in zip(got[1:], host[1:5]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("kind", ["terrain", "ties", "flat", "zeros", "wide", "tiny"])
@pytest.mark.parametrize("n,batch", [(1, 4), (33, 8), (511, 128), (4096, 1024), (4097, 1020),
                                     (70_003, 10240)])
def test_upload_equals_host_encoder(cuda_lib, n, batch, kind):
    xyz, rgba = _cloud(kind, n)
    for keep in (False, True):
        with pcr.Context(0, batch_size=batch, flags=pcr.PC_CFG_KEEP_ORDER if keep else 0) as ctx:
            for colours in (rgba, None):
                host = pcr.pc_encode(xyz, colours, batch, flags=pcr.PC_ENCODE_KEEP_ORDER if keep else 0)
                cloud = ctx.upload(xyz, colours)
                _same(ctx, cloud, host)
                pcr.pc_release_cloud(ctx.h, cloud)


def test_upload_of_a_million_points(cuda_lib):
    xyz, rgba = _cloud("terrain", 1_500_001)
    with pcr.Context(0) as ctx:
        _same(ctx, ctx.upload(xyz, rgba), pcr.pc_encode(xyz, rgba))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("at", [0, 4000, 9999])
def test_upload_refuses_what_the_host_encoder_refuses(cuda_lib, bad, at):
    xyz, rgba = _cloud("ties", 10_000)
    xyz[at, at % 3] = bad
    with pcr.Context(0) as ctx:
        with pytest.raises(pcr.PCError) as e:
            ctx.upload(xyz, rgba)
        assert e.value.status == pcr.PC_EINVAL
        assert pcr.pc_cloud_get_info(ctx.h, ctx.upload(xyz[:0], rgba[:0])).n_points == 0
