"""Power-of-two scales of the bf16 and e4m3 columns: the smallest 2^e that holds the largest
element, for significands on both sides of the format's and exponents over the whole range."""
import math

import pytest

from gpu_common import need_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt,fmax", [("bf16", 1.0), ("e4m3", 448.0)])
def test_scale_is_the_smallest_power(fmt, fmax):
    torch, cb = need_gpu()
    v = to_dev(torch, [0.0, 0.25])
    for e in (-1074, -1060, -1022, -1021, -300, -140, -127, -126, -119, -118, -117, -20, -9, -1, 0, 1, 9, 300, 1000):
        for m in (1.0, 1.0 + 2.0 ** -52, 1.5, 1.75 - 2.0 ** -52, 1.75, 1.75 + 2.0 ** -52, 2.0 - 2.0 ** -52):
            vmax = math.ldexp(m, e)
            k = -126
            while vmax > math.ldexp(fmax, k):
                k += 1
            assert cb.encode(fmt, v, vmax)[1] == math.ldexp(1.0, k), (fmt, m, e)
