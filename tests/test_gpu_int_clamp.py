"""Integer codes at and beyond the largest code: rounding to nearest, clamped to +-(2^(b-1) - 1)."""
import numpy as np
import pytest

from gpu_common import need_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt,mx,dt", [("i16", 32767, np.int16), ("i32", 2147483647, np.int32)])
def test_codes_clamp_at_the_ends(fmt, mx, dt):
    torch, cb = need_gpu()
    m = float(mx)
    k = np.array([0.0, 0.5, 1.5, 2.5, m - 1.5, m - 0.5, m, m + 0.25, m + 0.5, m + 1, m + 1.5, m + 2, 2 * m, 4294967296.0, 1e18,
                  1e300, np.inf])
    t = np.concatenate([k, -k])
    v = to_dev(torch, t)                      # vmax = mx: the scale is 1 and v * inv = v
    codes, scale = cb.encode(fmt, v, m)
    assert scale == 1.0
    got = codes.cpu().numpy().view(dt)[:t.size]
    assert np.array_equal(got.astype(np.int64), np.clip(np.rint(t), -m, m).astype(np.int64))
