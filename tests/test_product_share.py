"""hotrg_product_share: which steps contract by charge sectors, and how much of the product they execute."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(prec, dcut, steps, h, impure=0, charges=None, **kw):
    from paper_1911_12954_gb300 import HOTRG
    from paper_1911_12954_gb300.hotrg import OPT_CHARGES

    sched = [(i % 4, dcut) for i in range(steps)]
    g = HOTRG(batch=2, dcut_max=dcut, precision=prec, impure=impure, schedule=sched, **kw)
    g.init_tensor([1 / 6.62, 1 / 6.7], h)
    if charges is not None:
        g.set_option(OPT_CHARGES, charges)
    for mu, dc in sched:
        g.step(mu, dc)
    return g


@pytest.mark.parametrize("prec", ["fp64", "fp64oz", "fp32", "tf32x3", "fp16x3"])
@pytest.mark.parametrize("kw", [{}, dict(frac=0.3), dict(frac=0.16), dict(graphs=True)])
def test_runs_without_a_field_contract_by_sectors(prec, kw):
    """Every step of a run without a field, sliced workspaces and graphs included, and none of one with a field
    or with dropped charges."""
    full = _run(prec, 4, 5, 1e-300, impure=3)
    size = full.workspace.numel()
    kw = dict(workspace_bytes=int(size * kw["frac"])) if "frac" in kw else kw
    a = _run(prec, 4, 5, 0.0, impure=3, **kw)
    d = _run(prec, 4, 5, 0.0, impure=3, charges=16, **kw)
    for k in range(1, 6):
        for b in range(2):
            assert 0.2 < a.product_share(k, b) < 0.4, (k, b, a.product_share(k, b))
            assert full.product_share(k, b) == 1.0
            assert d.product_share(k, b) == pytest.approx(1.0, abs=1e-12)


def _parity(*q):
    """Indices of charge 0 and 1 among the multi-indices of legs with index charges q."""
    s = np.zeros(1, dtype=int)
    for v in q:
        s = (s[:, None] ^ v[None, :]).ravel()
    return np.array([np.sum(s == 0), np.sum(s == 1)], dtype=float)


@pytest.mark.parametrize("dcut", [3, 5])
@pytest.mark.parametrize("impure", [0, 3])
def test_share_counts_the_blocks(dcut, impure):
    """The share against a count over the charges read off the tensors' zeros: index i of a bond has the charge
    of index 0 where T[i, 0, 0, ...] is not zero, and index 0 is even."""
    for steps in range(2, 5):
        old, new = (_run("fp64", dcut, n, 0.0, impure=impure) for n in (steps - 1, steps))
        qs = []
        for g in (old, new):
            T = g.tensor(0, 0)
            qs.append([(T[tuple(slice(None) if leg == 2 * n else 0 for leg in range(8))] == 0.0).astype(int)
                       for n in range(4)])
        mu, c = (steps - 1) % 4, new.step_info(steps)["closing"]
        a, b = [n for n in range(4) if n not in (mu, c)]
        o, n = qs
        R = _parity(n[a], n[b], o[c], o[c], o[mu])
        K = _parity(o[a], o[b], o[a], o[b], o[mu])

        def part(pa, par):
            return sum(R[q] * R[q ^ par] * K[q ^ pa] for q in range(2))

        parts = [part(0, 0)] + ([part(1, 1), part(0, 1), part(0, 0), part(0, 0)] if impure else [])
        want = sum(parts) / (len(parts) * R.sum() ** 2 * K.sum())
        assert new.product_share(steps, 0) == pytest.approx(want, rel=1e-12)
