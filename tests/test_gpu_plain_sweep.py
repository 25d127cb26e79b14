"""FP64 storage at the sizes where its kernels have edges: boxes whose site count leaves a ragged
last block of the index-order sweep, particles of the smallest radius, boundary-site counts just
below and above one and two gathers of the ordered sums (128 entries), particles touching equilibrium
and no-slip faces, with and without a body force. Every operation is the oracle's, in its order, so
the results must agree to the last bits (1e-12 relative, as the other FP64 tests)."""
import numpy as np
import pytest

import oracle as O
from paper_1105_2904_gb300 import lbmp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1105_2904_gb300 import build as B
    B.build()
    O.build()


CASES = [
    dict(lattice=O.D3Q19, dims=(9, 8, 8), r=[1.5], walls=(0, 0, 0), eq={}, F=0.0),
    dict(lattice=O.D3Q19, dims=(33, 17, 11), r=[2.5, 1.5], walls=(0, 1, 0), eq={}, F=1e-5),
    dict(lattice=O.D3Q19, dims=(31, 29, 27), r=[3.3, 3.5, 3.7], walls=(0, 0, 0), eq={}, F=1e-5),
    dict(lattice=O.D3Q19, dims=(30, 20, 21), r=[4.5, 3.0], walls=(1, 0, 0), eq={0: (0.01, 0.0, 0.0), 1: (0.01, 0.0, 0.0)},
         F=0.0),
    dict(lattice=O.D2Q9, dims=(67, 45, 1), r=[12.0, 1.5], walls=(0, 1, 0), eq={2: (0.0, 0.0, 0.0)}, F=0.0),
    dict(lattice=O.D2Q9, dims=(128, 64, 1), r=[20.0], walls=(0, 0, 0), eq={}, F=1e-6),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c["dims"])))
def test_fp64_matches_oracle(case):
    nx, ny, nz = case["dims"]
    kw = dict(body_force=(case["F"], 0.0, 0.0), walls=case["walls"], gravity=(0.0, -1e-4, 0.0), equilibrium_faces=case["eq"],
              body_force_on_particles=case["F"] != 0.0)
    g = lbmp.Simulation(case["lattice"], nx, ny, nz, 0.7, precision="fp64", **kw)
    o = O.OracleSim(case["lattice"], nx, ny, nz, 0.7, **kw)
    c = np.zeros((len(case["r"]), 3))
    x = 0.0
    for k, r in enumerate(case["r"]):  # side by side along x, the first touching the -x and -y faces
        c[k] = (x + r - 0.5, r - 0.5 + 0.3 * k, 0.37 * nz if nz > 1 else 0.0)
        x += 2.0 * r + 0.6
    v = np.tile([0.03, 0.02, -0.025 if nz > 1 else 0.0], (len(c), 1))
    om = np.tile([0.0 if nz == 1 else 0.01, 0.0 if nz == 1 else -0.02, 0.02], (len(c), 1))
    for s in (g, o):
        s.add_particles(c, case["r"], np.full(len(c), 1.7), v, om)
    for n in (1, 1, 45):
        g.step(n)
        o.step(n)
        np.testing.assert_array_equal(g.get_tags(), o.get_tags())
        fg, fo = g.get_f(), o.get_f()
        assert np.max(np.abs(fg - fo)) <= 1e-12 * np.max(np.abs(fo))
        pg, po = g.get_particles(), o.get_particles()
        for q in po:
            assert np.max(np.abs(pg[q] - po[q])) <= 1e-12 * max(np.max(np.abs(po[q])), 1e-300), q
    g.close()
