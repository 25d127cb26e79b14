"""The particle phase around the sizes where its form changes: up to 1024 particles two launches with
a cluster, beyond one launch per phase; contact grids one, two, three and more cells wide, periodic
and walled; owner-map updates in one launch up to 262144 template entries; many particles crossing
site boundaries and colliding in every step. FP64 storage evaluates the oracle's operations in its
order, so particles and owner maps must agree to 1e-12 relative and exactly; FP32 within the 1e-4 of
the largest force that the other record tests use."""
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


CASES = [
    ("2d_1024", O.D2Q9, (330, 310, 1), 1024, 1.5, (0, 0, 0), 40),
    ("2d_1025_walls", O.D2Q9, (330, 310, 1), 1025, 1.5, (1, 1, 0), 40),
    ("3d_cells_1_2_3", O.D3Q19, (18, 26, 38), 14, 3.0, (0, 0, 0), 40),
    ("3d_walls", O.D3Q19, (19, 27, 39), 10, 3.0, (1, 0, 1), 40),
    ("2d_one_cell", O.D2Q9, (17, 60, 1), 5, 4.0, (0, 0, 0), 40),
    ("3d_entries_above", O.D3Q19, (110, 96, 90), 290, 6.0, (0, 0, 0), 4),
]


def _pair(case, precision):
    name, lattice, (nx, ny, nz), n, r, walls, steps = case
    D = 2 if lattice == O.D2Q9 else 3
    c, rad = W.rsa_centers((nx, ny, nz)[:D], n, r, seed=5, min_gap=0.3, walls=walls)
    v = np.clip(W.gaussian_velocities(n, 0.12, 6, D), -0.4, 0.4)
    om = np.zeros((n, 3))
    om[:, 2] = 0.02
    kw = dict(body_force=(1e-6, 0.0, 0.0), walls=walls, gap=0.4)
    g = lbmp.Simulation(lattice, nx, ny, nz, 0.8, precision=precision, **kw)
    o = O.OracleSim(lattice, nx, ny, nz, 0.8, **kw)
    for s in (g, o):
        s.add_particles(c, rad, np.full(n, 8.0), v, om)
    return g, o, steps


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_fp64_matches_oracle(case):
    g, o, steps = _pair(case, "fp64")
    for n in (1, steps - 1):
        g.step(n)
        o.step(n)
        np.testing.assert_array_equal(g.get_tags(), o.get_tags())
        pg, po = g.get_particles(), o.get_particles()
        for q in po:
            assert np.max(np.abs(pg[q] - po[q])) <= 1e-12 * np.max(np.abs(po[q])), q
        assert np.max(np.abs(g.get_orientations() - o.get_orientations())) <= 1e-13
    fg, fo = g.get_f(), o.get_f()
    assert np.max(np.abs(fg - fo)) <= 1e-12 * np.max(np.abs(fo))
    g.close()


@pytest.mark.parametrize("case", CASES[2:5], ids=[c[0] for c in CASES[2:5]])
@pytest.mark.parametrize("streaming", ["pull", "inplace"])
def test_fp32_forces_match_oracle(case, streaming):
    name, lattice, dims, n, r, walls, steps = case
    _, o, _ = _pair(case, "fp64")
    g, _, _ = _pair(case, "fp32")
    if streaming == "inplace":
        g.close()
        g = lbmp.Simulation(lattice, *dims, 0.8, body_force=(1e-6, 0.0, 0.0), precision="fp32", walls=walls, gap=0.4,
                            streaming="inplace")
        D = 2 if lattice == O.D2Q9 else 3
        c, rad = W.rsa_centers(dims[:D], n, r, seed=5, min_gap=0.3, walls=walls)
        om = np.zeros((n, 3))
        om[:, 2] = 0.02
        g.add_particles(c, rad, np.full(n, 8.0), np.clip(W.gaussian_velocities(n, 0.12, 6, D), -0.4, 0.4), om)
    worst = 0.0
    scale = 0.0
    for _ in range(20):
        g.step(1)
        o.step(1)
        fg, fo = g.get_particles()["force"], o.get_particles()["force"]
        scale = max(scale, np.max(np.abs(fo)))
        worst = max(worst, np.max(np.abs(fg - fo)))
    assert worst <= 1e-4 * scale
    np.testing.assert_array_equal(g.get_tags(), o.get_tags())
    g.close()
