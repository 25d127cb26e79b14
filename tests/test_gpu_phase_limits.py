"""The particle phase on both sides of every limit that changes its form, where the launches per phase
run: batches with a cell just above a limit beside a small, a walled and moving-walled, and an empty
cell, bit for bit the cells stepped alone (the batch changes how the work is launched, not what is
computed); and single contexts above the limits in the reduced storages, pull and in-place, against the
FP64 oracle with the bars of the other sweep tests (FP32 1e-5 of max|u| and 1e-4 of max|F|; FP16 2e-3
and 2e-2). Particles are fast enough that many shifts change in the steps taken."""
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


# lattice, first cell's dims, particles, radius
BATCHES = {
    "3d_256": (O.D3Q19, (57, 60, 62), 256, 2.0),
    "3d_257": (O.D3Q19, (57, 60, 62), 257, 2.0),
    "3d_entries_above": (O.D3Q19, (113, 104, 100), 240, 6.6),
    "2d_1025": (O.D2Q9, (330, 310, 1), 1025, 1.5),
    "2d_contact_cells_above": (O.D2Q9, (645, 642, 1), 200, 1.5),
}


def _particles(lattice, dims, n, r, walls, seed):
    D = 2 if lattice == O.D2Q9 else 3
    c, rad = W.rsa_centers(dims[:D], n, r, seed=seed, min_gap=0.3, walls=walls)
    v = np.clip(W.gaussian_velocities(n, 0.1, seed + 1, D), -0.3, 0.3)
    return c, rad, np.full(n, 8.0), v


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("walls", [(0, 1, 0), (0, 0, 0)], ids=["walls", "periodic"])
@pytest.mark.parametrize("name", list(BATCHES))
def test_batch_is_bitwise_its_cells(name, walls, precision):
    lattice, big, n, r = BATCHES[name]
    d2 = lattice == O.D2Q9
    dims = [big, (33, 26, 1 if d2 else 24), (20, 22, 1 if d2 else 18), (24, 20, 1 if d2 else 20)]
    parts = [_particles(lattice, big, n, r, walls, 5), _particles(lattice, dims[1], 3, 2.0, walls, 7), None,
             _particles(lattice, dims[3], 1, 2.0, walls, 9)]
    kw = dict(precision=precision, walls=walls, gap=0.3)
    b = lbmp.Batch(lattice, dims, [0.8] * 4, [(1e-5, 0.0, 0.0)] * 4, **kw)
    for k in (0, 1, 3):
        b.add_particles(k, *parts[k])
    if walls[1]:
        b.cell(1).set_wall_velocity(3, (0.03, 0.0, 0.0))
    b.set_tuning(order=1, steps_per_graph=3)
    b.step(8)
    b.synchronize()
    for k, d in enumerate(dims):
        s = lbmp.Simulation(lattice, *d, 0.8, body_force=(1e-5, 0.0, 0.0), **kw)
        s.set_sweep_shape(0)
        if k == 1 and walls[1]:
            s.set_wall_velocity(3, (0.03, 0.0, 0.0))
        if parts[k] is not None:
            s.add_particles(*parts[k])
        s.step(8)
        c = b.cell(k)
        np.testing.assert_array_equal(c.get_f(), s.get_f())
        if parts[k] is not None:
            np.testing.assert_array_equal(c.get_tags(), s.get_tags())
            pb, ps = c.get_particles(), s.get_particles()
            for q in ps:
                np.testing.assert_array_equal(pb[q], ps[q])
        s.close()
    b.close()


SINGLES = [
    ("2d_1025_walls", O.D2Q9, (330, 310, 1), 1025, 1.5, (1, 1, 0)),
    ("3d_entries_above", O.D3Q19, (110, 96, 90), 290, 6.0, (0, 0, 0)),
]


@pytest.mark.parametrize("precision,bar_u,bar_f", [("fp32", 1e-5, 1e-4), ("fp16", 2e-3, 2e-2)])
@pytest.mark.parametrize("streaming", ["pull", "inplace"])
@pytest.mark.parametrize("case", SINGLES, ids=[c[0] for c in SINGLES])
def test_above_the_limits_matches_oracle(case, streaming, precision, bar_u, bar_f):
    name, lattice, dims, n, r, walls = case
    parts = _particles(lattice, dims, n, r, walls, 5)
    kw = dict(body_force=(1e-6, 0.0, 0.0), walls=walls, gap=0.3)
    o = O.OracleSim(lattice, *dims, 0.8, **kw)
    g = lbmp.Simulation(lattice, *dims, 0.8, precision=precision, streaming=streaming, **kw)
    for s in (o, g):
        s.add_particles(*parts)
    before = o.get_tags().copy()
    for steps in (3, 2):  # both parities of the in-place layout
        o.step(steps)
        g.step(steps)
        np.testing.assert_array_equal(g.get_tags(), o.get_tags())
        _, uo = o.get_fields()
        _, ug = g.get_fields()
        assert np.max(np.abs(ug - uo)) <= bar_u * np.max(np.abs(uo))
        fo = o.get_particles()["force"]
        assert np.max(np.abs(g.get_particles()["force"] - fo)) <= bar_f * np.max(np.abs(fo))
    assert np.any(before != o.get_tags())
    g.close()


# A cell of a batch has one block for its contacts where a single context has a cluster, so the
# launches per phase take over at fewer particles (measured: between 200 and 300 a cell).
@pytest.mark.parametrize("n,few", [(256, True), (257, False)])
def test_batch_of_many_particles_a_cell_takes_the_launches_per_phase(n, few):
    parts = _particles(O.D3Q19, (57, 60, 62), n, 2.0, (0, 0, 0), 5)
    b = lbmp.Batch(O.D3Q19, [(57, 60, 62), (20, 20, 20)], [0.8] * 2, [(0.0, 0.0, 0.0)] * 2, precision="fp32", gap=0.3)
    b.add_particles(0, *parts)
    # sweep, sums, contacts and re-marking; or the sweep and at least one launch per phase
    assert (b.info()["launches_per_step"] == 4) == few
    b.close()
