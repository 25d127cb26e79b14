"""Sweeps in index order (one site per thread, used where 128-site row tiles would leave lanes idle):
row lengths that fill tiles badly, odd and even, boxes smaller than a block or with a ragged last one,
walls and moving walls, pull and in-place streaming, and batches whose cells take either form. A
site's arithmetic does not depend on the thread it runs on, so the oracle's bars of the other sweep
tests hold (FP32 1e-5 of max|u| and 1e-4 of max|F|; FP16 2e-3 and 2e-2), and a batch gives the bits
of its cells stepped alone, whatever its tile widths and order."""
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


BOXES = [
    (O.D3Q19, (9, 8, 8), (0, 0, 0)),
    (O.D3Q19, (9, 9, 11), (0, 0, 1)),
    (O.D3Q19, (129, 9, 8), (0, 1, 0)),
    (O.D3Q19, (115, 8, 9), (1, 0, 0)),     # just below nine tenths of a tile
    (O.D3Q19, (117, 8, 9), (0, 0, 0)),     # just above
    (O.D2Q9, (131, 9, 1), (0, 1, 0)),
    (O.D2Q9, (10, 10, 1), (0, 0, 0)),      # less than one block
]


def _sim(cls, box, **kw):
    lattice, (nx, ny, nz), walls = box
    two_d = nz == 1
    s = cls(lattice, nx, ny, nz, 0.8, body_force=(1e-5, 0.0, 0.0), walls=walls,
            wall_velocity={3: (0.02, 0.0, 0.0)} if walls[1] else {}, **kw)
    c = np.array([[nx / 2 + 0.2, ny / 2 - 0.1, 0.0 if two_d else nz / 2 + 0.3]])
    s.add_particles(c, [1.9], [1.5], np.array([[0.03, 0.01, 0.0 if two_d else -0.02]]), np.array([[0.0, 0.0, 0.02]]))
    return s


@pytest.mark.parametrize("precision,bar_u,bar_f", [("fp32", 1e-5, 1e-4), ("fp16", 2e-3, 2e-2)])
@pytest.mark.parametrize("streaming", ["pull", "inplace"])
@pytest.mark.parametrize("box", BOXES, ids=lambda b: "x".join(map(str, b[1])))
def test_ragged_boxes_match_oracle(box, streaming, precision, bar_u, bar_f):
    o = _sim(O.OracleSim, box)
    g = _sim(lbmp.Simulation, box, precision=precision, streaming=streaming)
    g.set_sweep_shape(0)
    for n in (31, 10):  # both parities of the in-place layout
        o.step(n)
        g.step(n)
        np.testing.assert_array_equal(g.get_tags(), o.get_tags())
        _, uo = o.get_fields()
        _, ug = g.get_fields()
        assert np.max(np.abs(ug - uo)) <= bar_u * np.max(np.abs(uo))
        fo = o.get_particles()["force"]
        assert np.max(np.abs(g.get_particles()["force"] - fo)) <= bar_f * np.max(np.abs(fo))
    g.close()


@pytest.mark.parametrize("order", [0, 1, 2])
@pytest.mark.parametrize("widths", [None, [32, 64, 32, 128]], ids=["128", "mixed"])
def test_batch_of_both_forms_gives_its_cells_bits(widths, order):
    dims = [(33, 17, 12), (64, 12, 11), (128, 16, 9), (21, 20, 19)]
    b = lbmp.Batch(O.D3Q19, dims, [0.7] * 4, [(1e-5, 0.0, 0.0)] * 4, precision="fp32")
    for k, d in enumerate(dims):
        b.add_particles(k, np.array([[d[0] / 2, d[1] / 2, d[2] / 2]]), [2.2], [1.4], np.array([[0.03, -0.02, 0.01]]))
    b.set_tuning(tile_width=widths, order=order, steps_per_graph=3)
    b.step(20)
    b.synchronize()
    for k, d in enumerate(dims):
        s = lbmp.Simulation(O.D3Q19, *d, 0.7, body_force=(1e-5, 0.0, 0.0), precision="fp32")
        s.set_sweep_shape(0)
        s.add_particles(np.array([[d[0] / 2, d[1] / 2, d[2] / 2]]), [2.2], [1.4], np.array([[0.03, -0.02, 0.01]]))
        s.step(20)
        np.testing.assert_array_equal(b.cell(k).get_f(), s.get_f())
        s.close()
    assert b.info()["tiles"] == len(lbmp.lbm_schedule_tiles(dims, widths, order))
    b.close()
