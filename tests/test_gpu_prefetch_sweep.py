"""FP32 two-site sweep with rows prefetched into L2 (boxes of at least 2^20 sites holding particles):
ny not a multiple of the block's four rows, so the last group of a plane is short, and rows whose
prefetch starts off a 16-byte boundary; periodic and walled, 2D and 3D. Against the FP64 oracle with the
FP32 bars of the other sweep tests (1e-5 of max|u|, 1e-4 of max|F|)."""
import numpy as np
import pytest

import oracle as O
from paper_1105_2904_gb300 import lbmp
from paper_1105_2904_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1105_2904_gb300 import build as B
    B.build()
    O.build()


@pytest.mark.parametrize("walls", [(0, 0, 0), (0, 1, 0)], ids=["periodic", "walls"])
@pytest.mark.parametrize("lattice,dims,r", [(O.D3Q19, (130, 91, 93), 5.0), (O.D2Q9, (1026, 1027, 1), 9.0)], ids=["3d", "2d"])
def test_prefetched_rows_match_oracle(lattice, dims, r, walls):
    D = 2 if lattice == O.D2Q9 else 3
    N = dims[0] * dims[1] * dims[2]
    n = int(0.12 * N / (np.pi * r * r if D == 2 else 4.0 / 3.0 * np.pi * r ** 3))
    c, rad = W.rsa_centers(dims[:D], n, r, seed=3, min_gap=0.5, walls=walls)
    v = np.clip(W.gaussian_velocities(n, 0.03, 4, D), -0.1, 0.1)
    kw = dict(body_force=(1e-5, 0.0, 0.0), walls=walls, gap=0.5)
    o = O.OracleSim(lattice, *dims, 0.8, **kw)
    g = lbmp.Simulation(lattice, *dims, 0.8, precision="fp32", **kw)
    for s in (o, g):
        s.add_particles(c, rad, np.full(n, 2.0), v)
        s.step(6)
    np.testing.assert_array_equal(g.get_tags(), o.get_tags())
    _, uo = o.get_fields()
    _, ug = g.get_fields()
    assert np.max(np.abs(ug - uo)) <= 1e-5 * np.max(np.abs(uo))
    fo = o.get_particles()["force"]
    assert np.max(np.abs(g.get_particles()["force"] - fo)) <= 1e-4 * np.max(np.abs(fo))
    g.close()
