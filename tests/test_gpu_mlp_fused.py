"""Closure network at the edges of the fused kernels' tiles: layer widths around 1, 8 and 16, one
layer and eight, row counts around the 16-row blocks, the 32-row ranges of the weight gradients and
the 256-row sums, and a network just too large for the fused form. Against the FP64 oracle with
bfloat16 emulation, with the bars of the other network tests (FP32 accumulation and rare bfloat16
rounding flips: 1e-2 of the largest entry, loss 1e-3); a training step is bit for bit the separate
gradient and Adam calls."""
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


SIZES = [[1, 1], [16, 8], [17, 15, 1], [259, 128, 128, 6], [24, 9, 16, 7, 8, 33, 5, 12, 3], [600, 430, 12]]


def _data(sizes, rows, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    p = M.init_params(sizes, seed)
    for layer in p:
        layer[0] = layer[0].astype(np.float32).astype(np.float64)
        layer[1] = g.normal(0, 0.2, layer[1].shape).astype(np.float32).astype(np.float64)
    X = g.normal(0, 1, (rows, sizes[0])).astype(np.float32)
    T = g.normal(0, 1, (rows, sizes[-1])).astype(np.float32)
    net = lbmp.MLP(sizes)
    net.set_params(p)
    return p, X, T, net, torch.tensor(X, device="cuda"), torch.tensor(T, device="cuda")


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-6))


@pytest.mark.parametrize("rows", [1, 15, 17, 129, 530])
@pytest.mark.parametrize("sizes", SIZES, ids=lambda s: "-".join(map(str, s)))
def test_forward_gradients_and_training(sizes, rows):
    p, X, T, net, x, t = _data(sizes, rows, 31 + rows)
    Xd, Td = X.astype(np.float64), T.astype(np.float64)
    Yr, _ = M.forward(p, Xd, bf16=True)
    assert _rel(net.forward(x).cpu().double().numpy(), Yr) <= 1e-2
    lr_, gr = M.loss_and_grads(p, Xd, Td, bf16=True)
    # all rows as one minibatch: training takes the same gradients, in another order of the rows
    losses = net.train(x, t, batch=rows, epochs=1, lr=1e-3, seed=4)
    for loss, gg in ((losses[0], net.grads()), (None, None)):
        if loss is None:
            net.set_params(p)
            loss = net.loss_grad(x, t)
            gg = net.grads()
        assert abs(loss - lr_) <= 1e-3 * lr_
        for l in range(len(sizes) - 1):
            assert _rel(gg[l][0], gr[l][0]) <= 1e-2, ("W", l)
            assert _rel(gg[l][1], gr[l][1]) <= 1e-2, ("b", l)
    net.close()


@pytest.mark.parametrize("sizes", SIZES, ids=lambda s: "-".join(map(str, s)))
def test_training_step_is_the_separate_calls(sizes):
    p, _, _, a, x, t = _data(sizes, 1, 5)
    b = _data(sizes, 1, 5)[3]
    for _ in range(3):
        a.train(x, t, batch=1, epochs=1, lr=1e-2)
        b.loss_grad(x, t)
        b.adam_step(1e-2)
    for (wa, ba), (wb, bb) in zip(a.params(), b.params()):
        np.testing.assert_array_equal(wa, wb)
        np.testing.assert_array_equal(ba, bb)
    np.testing.assert_array_equal(a.forward(x).cpu().numpy(), b.forward(x).cpu().numpy())
    a.close()
    b.close()
