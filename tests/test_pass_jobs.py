"""First half-contraction passes of both sides in one launch: the small form (one temperature at a time) and,
from four blocks per SM on, the form with a call for each job (the whole batch) give the same bits."""

import pytest

from workloads import decaying_tensor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16x3"])
@pytest.mark.parametrize("dims,mu,dcut,batch", [
    ((5, 5, 5, 2), 3, 4, 8),       # 49 blocks a job: 98 in all alone, 784 together
    ((3, 4, 2, 5), 1, 3, 48),      # odd and even legs, some 20 blocks alone
])
def test_small_and_large_launches_agree(prec, dims, mu, dcut, batch):
    from paper_1911_12954_gb300 import HOTRG

    out = []
    for group in (1, 0):
        g = HOTRG(batch=batch, dcut_max=5, precision=prec, schedule=[(mu, dcut)], dims0=dims, group=group)
        for b in range(batch):
            g.set_tensor(decaying_tensor(5 + b % 3, dims, 0.7), b)
        g.step(mu, dcut)
        assert g.step_info(1)["group"] == (1 if group else batch)
        out.append([g.tensor(0, b).tobytes() for b in range(batch)])
    assert out[0] == out[1]
