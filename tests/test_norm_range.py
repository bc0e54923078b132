"""ln c of a step whose coarse tensor is tiny: the norm of FP32 tensors over FP32's whole range."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "tf32x3"])
@pytest.mark.parametrize("eps", [1e-12, 1e-18, 1e-20, 1e-21, 1e-22, 1e-24, 1e-30])
def test_ln_c_of_a_tiny_coarse_tensor(precision, eps):
    """T = e0 x e1 x R + eps e1 x e0 x R on the legs (mu, mu'): of order 1, but the bond along mu joins
    the two terms, so every entry of T' is of order eps (squares down to 1e-60). The cut keeps every column,
    so ||T'|| is the norm of the joined pair, whatever the isometries. Relative error of an entry: about 60
    FP32 roundings (3.6e-6) and, for the tf32 pairs, 2^-21 of either operand: 1e-5 on ln c."""
    from paper_1911_12954_gb300 import HOTRG

    R = np.random.default_rng(2).uniform(0.5, 1.5, (2,) * 6)
    T = np.zeros((2,) * 8)
    T[0, 1], T[1, 0] = R, eps * R
    T /= np.linalg.norm(T)
    want = np.log(np.linalg.norm(np.tensordot(T, T, axes=(1, 0))))
    g = HOTRG(batch=1, dcut_max=4, precision=precision, schedule=[(0, 4)], dims0=(2, 2, 2, 2))
    g.set_tensor(T)
    g.step(0, 4)
    g.x_indicator()                          # raises if the norm was found not finite or zero
    assert abs(g.step_info(1)["ln_c"] - want) < 1e-5
    assert np.linalg.norm(g.tensor()) == pytest.approx(1.0, abs=1e-5)


@pytest.mark.parametrize("eps", [1e-36, 1e-37])
def test_ln_c_with_subnormal_entries(eps):
    """The same with entries of T' below FP32's normal range (eps / 100 of 2^-149 = 1.4e-45): 60 roundings of
    half a quantum are 3e-5 of such an entry, 1e-4 on ln c."""
    from paper_1911_12954_gb300 import HOTRG

    R = np.random.default_rng(2).uniform(0.5, 1.5, (2,) * 6)
    T = np.zeros((2,) * 8)
    T[0, 1], T[1, 0] = R, eps * R
    T /= np.linalg.norm(T)
    want = np.log(np.linalg.norm(np.tensordot(T, T, axes=(1, 0))))
    g = HOTRG(batch=1, dcut_max=4, precision="fp32", schedule=[(0, 4)], dims0=(2, 2, 2, 2))
    g.set_tensor(T)
    g.step(0, 4)
    assert abs(g.step_info(1)["ln_c"] - want) < 1e-4
