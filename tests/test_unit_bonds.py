"""Bonds of one index whose charge is odd: steps without a field after a cut to 1, with the bonds' charges
relabelled (OPT_CHARGES), against the same steps without."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SCHED = [(0, 3), (1, 1), (2, 4), (3, 3), (0, 4)]     # bonds of 1, 3, 1, 1 after two steps


def _run(prec, charges, stop):
    from paper_1911_12954_gb300 import HOTRG
    from paper_1911_12954_gb300.hotrg import OPT_CHARGES

    g = HOTRG(batch=1, dcut_max=4, precision=prec, impure=3, schedule=SCHED)
    g.workspace.fill_(0xFF)             # NaN bit patterns: nothing unwritten may be read
    g.torch.cuda.synchronize()          # (a run with graphs has a stream of its own)
    g.init_tensor(1 / 6.65, 0.0)
    for i, (mu, dc) in enumerate(SCHED[:stop]):
        if i in charges:
            g.set_option(OPT_CHARGES, charges[i])
        g.step(mu, dc)
    return g


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-13), ("tf32x3", 3e-6)])
@pytest.mark.parametrize("at", [2, 3, 4])
@pytest.mark.parametrize("bits", [1, 2, 4, 8, 5, 9, 12, 15])
def test_relabelled_unit_bonds(prec, tol, at, bits):
    """The relabelling moves no zero: the step before which it is made gives the same tensors up to the order
    of sums (FP64: 1e-13 of the largest entry; tf32 pairs: 2^-21 of either operand and FP32 sums of at most
    144 terms, 3e-6) and the same discarded sums."""
    a, b = _run(prec, {at: bits}, at + 1), _run(prec, {}, at + 1)
    for which in range(3):
        x, y = a.tensor(which), b.tensor(which)
        assert np.max(np.abs(x - y)) <= tol * np.max(np.abs(y)), which
    ea, eb = np.array(a.step_info(at + 1)["eps"]), np.array(b.step_info(at + 1)["eps"])
    assert np.max(np.abs(ea - eb)) <= tol
