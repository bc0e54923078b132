"""FP32 and FP64 products on both sides of the line between small and large tiles."""

import numpy as np
import pytest

from workloads import decaying_tensor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,mu,dcut", [
    ((4, 4, 4, 3), 3, 4),      # M = N = 768, K = 768: 288 small tiles
    ((5, 5, 5, 2), 3, 4),      # M = N = 800, K = 1250: 325, ragged
    ((4, 4, 4, 4), 0, 4),      # M = N = 1024, K = 1024: 512, so 128 large ones
    ((5, 5, 5, 3), 3, 4),      # M = N = 1200, K = 1875: large ones, ragged
])
@pytest.mark.parametrize("batch", [1, 3])
def test_fp32_step_vs_fp64(dims, mu, dcut, batch):
    """3e-5 of the largest entry, the bound the FP32-storage steps have against FP64 ones."""
    from paper_1911_12954_gb300 import HOTRG

    out = []
    for prec in ("fp64", "fp32"):
        g = HOTRG(batch=batch, dcut_max=5, precision=prec, schedule=[(mu, dcut)], dims0=dims)
        for b in range(batch):
            g.set_tensor(decaying_tensor(5 + b, dims, 0.7), b)
        g.step(mu, dcut)
        out.append([g.tensor(0, b) for b in range(batch)])
    for x, y in zip(*out):
        assert np.abs(x - y).max() <= 3e-5 * np.abs(x).max()
