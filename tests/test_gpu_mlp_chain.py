"""Training over several minibatches, launched as an overlapping chain, is bit for bit the same minibatches
taken one call at a time (gradients, then Adam): the permutation is the library's (std::shuffle over
mt19937, from a host program), the batch's last 16-row block is partial, rows are left over, and there are
two epochs. A minibatch lost or taken twice, weights read too early or a step count off by one shows in
the bits. For the fused network and for one that runs layer by layer; repeated, for a race that needs luck."""
import shutil
import subprocess

import numpy as np
import pytest

from oracle import mlp_oracle as M
from paper_1105_2904_gb300 import lbmp

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

PROGRAM = r'''
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
int main(int, char** v)
{
    const int n = std::atoi(v[1]), epochs = std::atoi(v[2]);
    std::mt19937 rng((unsigned)std::atoi(v[3]));
    std::vector<int> perm(n);
    for (int e = 0; e < epochs; ++e) {
        for (int i = 0; i < n; ++i) perm[i] = i;
        std::shuffle(perm.begin(), perm.end(), rng);
        for (int i : perm) std::printf("%d ", i);
    }
}
'''


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1105_2904_gb300 import build as B
    B.build()


@pytest.mark.parametrize("sizes,batch", [([259, 128, 128, 6], 200), ([17, 40, 33, 5], 24), ([600, 430, 12], 200)],
                         ids=["closure", "small", "layers"])
def test_training_chain_is_the_separate_calls(tmp_path, sizes, batch):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not found")
    n, epochs, seed, lr = 3 * batch + 7, 2, 11, 1e-2
    src, exe = tmp_path / "perm.cc", tmp_path / "perm"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe), str(n), str(epochs), str(seed)], check=True, capture_output=True, text=True).stdout
    perms = np.array(out.split(), dtype=np.int64).reshape(epochs, n)
    g = np.random.Generator(np.random.PCG64(6))
    x = torch.tensor(g.normal(0, 1, (n, sizes[0])).astype(np.float32), device="cuda")
    t = torch.tensor(g.normal(0, 1, (n, sizes[-1])).astype(np.float32), device="cuda")
    p = M.init_params(sizes, 2)
    a, b = lbmp.MLP(sizes), lbmp.MLP(sizes)
    b.set_params(p)
    want = []
    for perm in perms:
        losses = []
        for k in range(n // batch):
            rows = torch.tensor(perm[k * batch:(k + 1) * batch], device="cuda")
            losses.append(b.loss_grad(x[rows].contiguous(), t[rows].contiguous()))
            b.adam_step(lr)
        want.append(sum(losses) / len(losses))
    for _ in range(3):
        a.set_params(p)
        losses = a.train(x, t, batch=batch, epochs=epochs, lr=lr, seed=seed)
        for (wa, ba), (wb, bb) in zip(a.params(), b.params()):
            np.testing.assert_array_equal(wa, wb)
            np.testing.assert_array_equal(ba, bb)
        assert np.max(np.abs(np.asarray(losses) - want)) <= 1e-12 * max(want)  # (64-bit sums of the same values)
    a.close()
    b.close()
