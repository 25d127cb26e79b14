"""Loss of the fused network over one warp's sums of 256 outputs, just beyond, over a ragged last sum, and
over many warps, called again after a larger call (the counter of finished warps is back at zero), against
the squared errors of the forward pass summed in 64 bits. A sum of 256 non-negative FP32 values by a tree
is off by at most eight roundings, 8 x 6e-8 < 1e-6, and the sums are added in 64 bits."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from paper_1105_2904_gb300 import lbmp

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1105_2904_gb300 import build as B
    B.build()


def test_loss_over_many_outputs():
    sizes = [12, 40, 64]
    net = lbmp.MLP(sizes)
    net.set_params(M.init_params(sizes, 3))
    g = np.random.Generator(np.random.PCG64(8))
    for rows in (15, 16, 17, 40, 1000, 4096, 16385, 16):
        x = torch.tensor(g.normal(0, 1, (rows, 12)).astype(np.float32), device="cuda")
        t = torch.tensor(g.normal(0, 1, (rows, 64)).astype(np.float32), device="cuda")
        want = float(((net.forward(x) - t).double() ** 2).mean())
        for loss in (net.loss_grad(x, t), net.loss_grad(x, t)):
            assert abs(loss - want) <= 1e-6 * want, rows
    net.close()
