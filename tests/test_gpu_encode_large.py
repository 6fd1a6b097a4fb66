"""pc_upload_cloud against the host encoder, bit for bit, where the device encoder's sort
takes its further steps: the scan over the tiles' sums works in rounds of 256 sums of 8
tiles of 4,096 points, so its second round starts at 8,388,609 points, and the points'
byte offsets pass 2^32 at 357,913,942."""
import numpy as np
import pytest

import paper_2204_01287_gb300 as pcr
import pcsynth as S

pytestmark = pytest.mark.gpu


def _same(n, flags):
    p = S.terrain_params(20000.0, 0.2, 5000)
    xyz, rgba = np.empty((n, 3), np.float32), np.empty(n, np.uint32)
    S.terrain(n, p, seed=11, out=(xyz, rgba))
    host = pcr.pc_encode(xyz, rgba, 10240, flags=pcr.PC_ENCODE_KEEP_ORDER if flags else 0)
    with pcr.Context(0, flags=flags) as ctx:
        cloud = ctx.upload(xyz, rgba)
        del xyz, rgba
        got = pcr.pc_cloud_download(ctx.h, cloud)
        assert got[0].tobytes() == host[0].tobytes()
        for a, b in zip(got[1:], host[1:5]):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("flags", [0, pcr.PC_CFG_KEEP_ORDER])
@pytest.mark.parametrize("n", [8_388_608, 8_388_609, 20_000_003])
def test_second_round_of_the_scan(cuda_lib, n, flags):
    _same(n, flags)


def test_offsets_past_four_gib(cuda_lib):
    _same(360_000_001, 0)
