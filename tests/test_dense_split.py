"""The fp16 operand planes of dense steps with odd legs (whole ranges of the summed index per block)
against the FP64 step of the same tensor."""

import numpy as np
import pytest

from workloads import decaying_tensor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,mu,dcut", [
    ((3, 3, 3, 3), 0, 3),      # one short panel, rows of 5 mod 8 values
    ((2, 2, 3, 2), 2, 2),      # ranges of 24 values, two row groups a side
    ((5, 5, 5, 2), 0, 9),      # 9 kept columns: the tile takes only part of the a2 range
    ((7, 7, 7, 2), 1, 3),      # several panels, one a2 each
    ((5, 2, 3, 4), 0, 6),      # odd direction, even transverse legs
    ((8, 8, 3, 3), 3, 5),      # contraction length 8
    ((9, 3, 9, 2), 1, 4),      # a leg past the range: the general form
])
@pytest.mark.parametrize("maxnorm", [True, False])
def test_odd_legs_vs_fp64(dims, mu, dcut, maxnorm):
    """3e-5 of the largest entry, the bound the FP32-storage steps have against the oracle (FP32 tensors and
    isometries, 22-bit operands)."""
    from paper_1911_12954_gb300 import HOTRG

    T = decaying_tensor(5, dims, 0.7)
    out = []
    for prec in ("fp64", "fp16x3"):
        g = HOTRG(batch=1, dcut_max=9, precision=prec, schedule=[(mu, dcut)], dims0=dims,
                  **({"maxnorm": maxnorm} if prec == "fp16x3" else {}))
        g.workspace.fill_(0xFF)        # NaN bit patterns: nothing unwritten may be read
        g.set_tensor(T)
        g.step(mu, dcut)
        out.append(g.tensor())
    assert np.abs(out[1] - out[0]).max() <= 3e-5 * np.abs(out[0]).max()
