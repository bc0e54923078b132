"""Runs without a field whose charges are dropped on the way (one sector, the dense product) against
the dense run: T, S and M, from the first step on and from a later one.

A field of 1e-300 gives the same site tensors bit for bit but takes the dense contraction."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DROP = 16
TOL = {"fp64": 1e-12, "fp64oz": 1e-9, "tf32x3": 2e-6, "fp16x3": 2e-6}   # on ln Z/V, as for the other sector runs


def _run(prec, dcut, steps, h, charges=None, **kw):
    """charges: {step: option value}, set before that step (0-based)."""
    from paper_1911_12954_gb300 import HOTRG
    from paper_1911_12954_gb300.hotrg import OPT_CHARGES

    sched = [(i % 4, dcut) for i in range(steps)]
    g = HOTRG(batch=2, dcut_max=dcut, precision=prec, impure=3, schedule=sched, **kw)
    g.workspace.fill_(0xFF)             # NaN bit patterns: nothing unwritten may be read
    g.torch.cuda.synchronize()          # (a run with graphs has a stream of its own)
    g.init_tensor([1 / 6.62, 1 / 6.7], h)
    for i, (mu, dc) in enumerate(sched):
        if charges and i in charges:
            g.set_option(OPT_CHARGES, charges[i])
        g.step(mu, dc)
    return g


@pytest.mark.parametrize("prec", ["fp64", "fp64oz", "tf32x3", "fp16x3"])
@pytest.mark.parametrize("dcut,steps,at", [(3, 6, 0), (4, 5, 0), (4, 6, 2), (5, 4, 3)])
def test_dropped_charges_give_the_dense_step(prec, dcut, steps, at):
    """ln Z/V, <sigma sigma> and the Frobenius norms of S and M (free of the isometries' signs) of a run that
    drops its charges before step `at`: those of the dense run, to the bounds of test_sectors.py; the norms
    to 20 times ln Z/V's (they are ratios of single tensors, not sums over the steps)."""
    a = _run(prec, dcut, steps, 0.0, {at: DROP})
    b = _run(prec, dcut, steps, 1e-300)
    assert np.max(np.abs(a.lnZ() - b.lnZ())) < TOL[prec]
    assert np.max(np.abs(a.energy()[1] - b.energy()[1])) < 20 * TOL[prec]
    for which in (1, 2):
        for e in range(2):
            x, y = np.linalg.norm(a.tensor(which, e)), np.linalg.norm(b.tensor(which, e))
            assert y > 1e-3 and abs(x - y) < 20 * TOL[prec], (which, e, x, y)


@pytest.mark.parametrize("kw", [dict(graphs=True), dict(group=1), dict(frac=0.3)])
def test_dropped_charges_under_graphs_groups_and_slices(kw):
    """The same in captured graphs, one temperature at a time and with a sliced workspace (FP64)."""
    full = _run("fp64", 4, 5, 0.0, {1: DROP})
    kw = dict(workspace_bytes=int(full.workspace.numel() * kw["frac"])) if "frac" in kw else kw
    a = _run("fp64", 4, 5, 0.0, {1: DROP}, **kw)
    for which in range(3):
        x, y = a.tensor(which, 1), full.tensor(which, 1)
        assert np.max(np.abs(x - y)) <= 1e-13 * np.max(np.abs(y)), which


def test_charge_option_is_refused_where_there_are_no_charges():
    from paper_1911_12954_gb300 import HotrgError

    with pytest.raises(HotrgError, match="ESTATE"):
        _run("fp64", 2, 1, 1e-5, {0: DROP})
    with pytest.raises(HotrgError, match="EINVAL"):
        _run("fp64", 2, 1, 0.0, {0: 32})
