"""Row counts that do not fill the fused network's blocks.

Loss of the fused network over one warp's sums of 256 outputs, just beyond, over a ragged last sum, and
over many warps, called again after a larger call (the counter of finished warps is back at zero), against
the squared errors of the forward pass summed in 64 bits. A sum of 256 non-negative FP32 values by a tree
is off by at most eight roundings, 8 x 6e-8 < 1e-6, and the sums are added in 64 bits.

Rows beyond the last of a 16-row block: a network whose hidden values overflow for an all-zero input but
not for the one real row has the finite gradients of that row (all products exact)."""
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


def test_rows_beyond_the_last_take_no_part():
    big = 2.0 ** 127
    net = lbmp.MLP([1, 1, 1, 1])
    # x = 1: hidden values 0 and 1; x = 0: 2^127 and infinity
    net.set_params([[np.array([[-big]]), np.array([big])], [np.array([[4.0]]), np.array([1.0])],
                    [np.array([[1.0]]), np.array([0.0])]])
    one = torch.ones(1, 1, device="cuda")
    assert net.loss_grad(one, 0.0 * one) == 1.0
    grads = [float(g.ravel()[0]) for layer in net.grads() for g in layer]
    assert grads == [0.0, 0.0, 0.0, 2.0, 2.0, 2.0]
    net.close()
