"""The contraction by Z2 charge sectors (no field) against the dense contraction and the oracle.

A field of 1e-300 gives the same site tensors bit for bit (exp(beta h) rounds to 1) but takes the
dense contraction, so the two paths can be compared on the same inputs: odd and even cuts, cuts
whose kept columns split unevenly between the charges, pure and impure tensors (S is odd under
the charge), groups of temperatures, sliced workspaces and captured graphs.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DENSE = 1e-300      # a field too small to change any entry
TOL = {"fp64": 1e-12, "fp64oz": 1e-9, "fp32": 2e-6, "tf32x3": 2e-6, "fp16x3": 2e-6}


def _run(prec, dcut, steps, h, impure=0, temps=(6.62, 6.7), **kw):
    from paper_1911_12954_gb300 import HOTRG

    sched = [(i % 4, dcut) for i in range(steps)]
    g = HOTRG(batch=len(temps), dcut_max=dcut, precision=prec, impure=impure, schedule=sched, **kw)
    g.workspace.fill_(0xFF)             # NaN bit patterns: nothing unwritten may be read
    g.init_tensor([1 / t for t in temps], h)
    for mu, dc in sched:
        g.step(mu, dc)
    out = [g.lnZ()]
    if impure:
        out += [g.energy()[1], g.magnetization()]
    return g, out


@pytest.mark.parametrize("prec", ["fp64", "fp64oz", "fp32", "tf32x3", "fp16x3"])
@pytest.mark.parametrize("dcut,steps", [(2, 9), (3, 8), (4, 7), (5, 5), (6, 4)])
def test_sector_runs_match_dense_runs(prec, dcut, steps):
    """ln Z/V of a run by sectors and of the dense run: equal to the mode's accuracy (FP64: the
    same terms in the same order but for the exact zeros, so rounding only)."""
    _, a = _run(prec, dcut, steps, 0.0)
    _, b = _run(prec, dcut, steps, DENSE)
    assert np.max(np.abs(a[0] - b[0])) < TOL[prec], (a, b)


@pytest.mark.parametrize("prec", ["fp64", "fp64oz", "tf32x3", "fp16x3"])
def test_sector_impure_runs(prec):
    """T, S and M: <sigma> is exactly zero by symmetry, <sigma sigma> that of the dense run."""
    _, a = _run(prec, 4, 6, 0.0, impure=3)
    _, b = _run(prec, 4, 6, DENSE, impure=3)
    assert np.max(np.abs(a[0] - b[0])) < TOL[prec]
    assert np.max(np.abs(a[1] - b[1])) < 20 * TOL[prec]
    assert np.all(a[2] == 0.0)


@pytest.mark.parametrize("mu", range(4))
@pytest.mark.parametrize("which", [0, 1, 2])
def test_sector_step_tensor_elementwise_fp64(mu, which):
    """Every entry of the coarse T, S and M after a step along each direction, FP64, uneven
    extents: 1e-13 of the largest entry off the dense step's, and exact zeros where the dense
    step has them."""
    from paper_1911_12954_gb300 import HOTRG

    sched = [(mu, 3), ((mu + 1) % 4, 5), ((mu + 3) % 4, 4)]
    out = []
    for h in (0.0, DENSE):
        g = HOTRG(batch=1, dcut_max=5, precision="fp64", impure=3, schedule=sched)
        g.init_tensor(1 / 6.65, h)
        for m, dc in sched:
            g.step(m, dc)
        out.append(g.tensor(which))
    assert np.max(np.abs(out[0] - out[1])) < 1e-13 * np.max(np.abs(out[1]))
    assert np.array_equal(out[0] == 0.0, out[1] == 0.0)


@pytest.mark.parametrize("prec", ["fp64", "fp16x3"])
def test_sector_slices_groups_and_graphs(prec):
    """One temperature at a time and captured graphs give the bits of the grouped, eager run;
    slices of the new a leg on both sides too in FP64 (the fp16 planes are scaled slice by slice,
    so there to the 1e-6 of the dense slicing test)."""
    ref, a = _run(prec, 4, 6, 0.0, impure=3)
    full = ref.workspace.numel()
    seen = set()
    for kw in (dict(group=1), dict(graphs=True), dict(workspace_bytes=int(full * 0.3)),
               dict(workspace_bytes=int(full * 0.16))):
        g, b = _run(prec, 4, 6, 0.0, impure=3, **kw)
        seen.add(g.step_info(6)["slices"])
        if prec == "fp64" or "workspace_bytes" not in kw:
            assert all(np.array_equal(x, y) for x, y in zip(a, b)), kw
            assert g.tensor(0, 1).tobytes() == ref.tensor(0, 1).tobytes()
        else:
            assert all(np.max(np.abs(x - y)) < 1e-6 for x, y in zip(a, b)), kw
    assert len(seen) > 1, seen


@pytest.mark.parametrize("impure", [0, 3])
def test_sector_split_statistics_count_every_entry(impure):
    """hotrg_split_stats over operands stored by sectors after the first step, whose operands are
    the dense step's bit for bit: the same counts, the exact zeros left out included."""
    a, _ = _run("fp16x3", 4, 1, 0.0, temps=(6.65,), impure=impure)
    b, _ = _run("fp16x3", 4, 1, DENSE, temps=(6.65,), impure=impure)
    assert a.split_stats() == b.split_stats()
