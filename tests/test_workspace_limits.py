"""Steps in workspaces that hold the contraction but not the isometry stage's ordinary space: many
temperatures at a small cut, one long leg among short ones, down to the least a step takes."""

import numpy as np
import pytest

from workloads import decaying_tensor

pytestmark = pytest.mark.gpu

# 3e-5 of the largest entry is the bound the FP32-storage steps have against FP64 ones; FP64: the Gram sums are
# taken in other chunks (1e-15 of their size) and the eigenvectors move by that over the gaps between eigenvalues
TOL = {"fp64": 1e-10, "fp32": 3e-5, "fp16x3": 3e-5}


def _step(prec, batch, dims, mu, dcut, **kw):
    from paper_1911_12954_gb300 import HOTRG

    g = HOTRG(batch=batch, dcut_max=max(*dims, dcut), precision=prec, schedule=[(mu, dcut)], dims0=dims, **kw)
    g.workspace.fill_(0xFF)                 # NaN bit patterns: nothing unwritten may be read
    g.torch.cuda.synchronize()
    for b in range(batch):
        g.set_tensor(decaying_tensor(5 + b % 3, dims, 0.7), b)
    g.step(mu, dcut)
    return g


@pytest.mark.parametrize("prec,batch,dims,mu,dcut,nbytes", [
    ("fp16x3", 32, (4, 4, 4, 4), 0, 4, 34202880),       # a batch's eigenproblems in several launches
    ("fp16x3", 32, (4, 4, 4, 4), 0, 4, 27912960),
    ("fp32", 32, (2, 1, 2, 9), 1, 2, 19642112),         # 81 x 81 matrices beside a tiny contraction
    ("fp16x3", 4, (12, 2, 2, 2), 1, 4, 14583040),
    ("fp16x3", 4, (12, 2, 2, 2), 1, 4, 6768640),        # 144 x 144, one matrix at a time, a one-sweep log
    ("fp32", 8, (16, 1, 1, 1), 1, 4, 79231488),
    ("fp32", 8, (16, 1, 1, 1), 1, 4, 31321088),         # 256 x 256: the matrix itself in the work space
    ("fp64", 1, (8, 2, 2, 2), 2, 4, 1178368),
    ("fp64", 2, (1, 1, 1, 1), 0, 2, 1 << 20),
])
def test_step_in_a_small_workspace(prec, batch, dims, mu, dcut, nbytes):
    a = _step(prec, batch, dims, mu, dcut, workspace_bytes=nbytes)
    b = _step(prec, batch, dims, mu, dcut)
    for e in {0, batch - 1}:
        assert abs(a.step_info(1, e)["ln_c"] - b.step_info(1, e)["ln_c"]) <= TOL[prec]
        x, y = a.tensor(0, e), b.tensor(0, e)
        assert np.max(np.abs(x - y)) <= TOL[prec] * np.max(np.abs(y)), e
