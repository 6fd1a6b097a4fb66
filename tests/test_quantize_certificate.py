"""The device encoder's quantization (encode.cu): a quotient by the rounded reciprocal,
added to 2^32, decides the whole part unless its fraction is the first or the last step
of 2^-20. Checked on the CPU in the same binary64 operations against the definition's
divide, at random quotients and at quotients next to whole numbers; with the first step
taken as certain too, the check must fail."""
import numpy as np
import pytest


def _cases(scale, n, seed):
    """Distances d in boxes of size s (binary64 and binary32 sizes) whose quotients are
    anywhere, or within a few roundings of a whole number."""
    r = np.random.default_rng(seed)
    size = np.exp2(r.uniform(-140, 127, n))
    size = np.where(r.random(n) < 0.5, size.astype(np.float32).astype(np.float64), size)
    d = size * r.random(n)
    whole = np.floor(r.uniform(0, scale, n))
    near = whole / scale * size
    near = near + np.spacing(near) * r.integers(-3, 4, n)
    d = np.where(r.random(n) < 0.7, near, d)
    top = r.random(n) < 0.01
    d[top] = size[top] * (1 + r.choice([0.0, 2.0 ** -24, -2.0 ** -53], int(top.sum())))
    return np.maximum(d, 0.0), size


@pytest.mark.parametrize("scale", [2.0 ** 21, 2.0 ** 30])
def test_certain_quotients_are_the_definitions(scale):
    certain = total = wrong = 0
    for seed in range(8):
        d, size = _cases(scale, 1_000_000, seed)
        exact = np.minimum(np.floor((scale * d) / size), scale - 1)
        t = d * (scale / size)
        bits = (t + 2.0 ** 32).view(np.uint64)
        fraction = (bits & np.uint64(0xFFFFF)).astype(np.int64)
        whole = np.minimum(((bits >> np.uint64(20)) & np.uint64(0xFFFFFFFF)).astype(np.float64), scale - 1)
        inside = (bits >> np.uint64(52)) == 1023 + 32
        sure = inside & (fraction >= 1) & (fraction <= 2 ** 20 - 2)
        assert np.array_equal(whole[sure], exact[sure])
        certain += int(sure.sum())
        total += len(d)
        loose = inside & (fraction <= 2 ** 20 - 2)
        wrong += int((whole[loose] != exact[loose]).sum())
    assert certain > 0.2 * total
    # a sum rounded up to a whole number; the last step is margin, since the two
    # quotients lie within 0.375 steps of each other
    assert wrong > 0
