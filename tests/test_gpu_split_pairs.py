"""FP64 codes split two at a time into FP32 pairs: every combination of value classes in the two
halves of a 16-byte chunk, through the basis update w - V c with one column."""
import itertools

import numpy as np
import pytest

from gpu_common import need_gpu, to_dev

pytestmark = pytest.mark.gpu

EDGE = [0.0, -0.0, 1.0, -2.0 + 2.0 ** -52, 2.0 ** -74, -(2.0 ** -74) * (1 + 2.0 ** -52), 2.0 ** -75 * (2 - 2.0 ** -52),
        2.0 ** -126, 2.0 ** -127, 1e-300, 5e-324, 1.0 + 2.0 ** -24, 1.0 + 2.0 ** -23, 1.0 + 2.0 ** -52, 2.0 ** 100 * 1.1,
        -(2.0 ** 120) * (2 - 2.0 ** -52)]


@pytest.mark.parametrize("entry", ["axpy", "dot"])
def test_pairs_of_value_classes(entry):
    torch, cb = need_gpu()
    rng = np.random.default_rng(5)
    v = np.array(list(itertools.product(EDGE, EDGE))).ravel()
    v = np.concatenate([v, rng.standard_normal(512) * 2.0 ** rng.integers(-90, 60, 512)])
    n = 4096
    x = np.zeros(n)
    x[:v.size] = v
    if entry == "axpy":
        w = torch.zeros(n, dtype=torch.float64, device="cuda")
        got = cb.basis_axpy("f64", "df32", n, torch.from_numpy(x[None]).cuda(), n, np.ones(1), -np.ones(1), w).cpu().numpy()
    else:                                     # one column per value, times a vector of ones
        m = 300
        pick = rng.permutation(v.size)[:m]
        cols = np.zeros((m, n))
        cols[np.arange(m), pick] = v[pick]
        got, x = cb.basis_dot("f64", "df32", n, torch.from_numpy(cols).cuda(), n, np.ones(m), to_dev(torch, np.ones(n))), v[pick]
    # hi + lo = x within 2^-48; below 2^-74 only hi is kept; the pair's sums round below 2^-48
    assert np.all(np.abs(got - x) <= 2.0 ** -47 * np.abs(x) + 2.0 ** -98)
