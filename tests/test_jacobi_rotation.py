"""The cosine of a Jacobi rotation as the eigensolver forms it: c = (1 + t^2)^(-1/2) from an FP32 start r
by the binomial series of (1 - e)^(-1/2) = 1 + e/2 + 3/8 e^2 + 5/16 e^3 + ..., 1 - e = (1 + t^2) r^2."""

import numpy as np
import pytest

L = np.longdouble


def _cosine(t, ulps):
    """t: FP32 tangents; ulps: error of the start in units in the last place (rsqrtf is within 2, and its
    argument, rounded to FP32, adds half of one to the root)."""
    t64 = t.astype(np.float64)
    x = 1.0 + t64 * t64                                   # the square is exact: one rounding, as the FMA
    r = (1 / np.sqrt(x)).astype(np.float32)
    r = (r + np.float32(ulps) * np.spacing(r)).astype(np.float64)
    e = (L(1) - L(1) * x * (r * r)).astype(np.float64)    # r * r is exact; extended product for the FMA
    return (L(1) * r + L(1) * (r * e) * (e * 0.375 + 0.5)).astype(np.float64), x


@pytest.mark.parametrize("ulps", [-3, -1, 0, 1, 3])
def test_cosine_to_fp64_accuracy(ulps):
    """Relative error below 2.5 2^-53: x rounds once (2^-54 on the root) and so does the result (2^-53 of a
    number below 1, 2^-52.5 relative to the smallest c, 2^-1/2); the series stops at 5/16 e^3 with |e| < 2^-20."""
    rng = np.random.default_rng(4)
    t = np.concatenate([2.0 ** rng.uniform(-61, 0, 200000), 1 - 2.0 ** rng.uniform(-24, -1, 20000), [0.0, 1.0],
                        rng.uniform(0, 1, 200000)]).astype(np.float32)
    c, x = _cosine(t, ulps)
    exact = 1 / np.sqrt(L(1) + L(1) * t.astype(np.float64) * t.astype(np.float64))
    assert np.max(np.abs((c - exact) / exact)) < 2.5 * 2.0 ** -53
    # the rotation's columns: c^2 + (c t)^2 = 1 to the same accuracy
    assert np.max(np.abs(L(1) * c * c * (L(1) + L(1) * t.astype(np.float64) ** 2) - 1)) < 5 * 2.0 ** -53
