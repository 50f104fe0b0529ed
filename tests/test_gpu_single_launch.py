"""The single-launch step against the graph of four kernels, bit for bit: tile
shapes (meshes narrower than a tile, two tiles a row, a last tile with one
column, one plane a tile and several), charges held in registers (up to 8 a
particle warp: 4864 on 152 SMs) and several passes over them, few steps and
more than one launch's worth, and the host loop's round trip."""
import numpy as np
import pytest

from paper_1309_7859_gb300 import inputs
from paper_1309_7859_gb300.inputs import EpsSpec

pytestmark = pytest.mark.gpu

TH = (1.0, 1.0)


def pair(mesh, n, precision, cell, self_mode=1):
    from paper_1309_7859_gb300.memd import Memd
    rng = np.random.default_rng(n + mesh[0])
    box = tuple(cell * N for N in mesh)
    eps = EpsSpec("vertices", 0, (), inputs.smooth_random_vertices(rng, mesh, 1.0))
    x, q = inputs.uniform_positions(rng, n, box), inputs.neutral_charges(rng, n)
    m, v = rng.uniform(0.5, 2.0, n), inputs.thermal_velocities(rng, n)
    out = []
    for e in ("single", "graph"):
        g = Memd(mesh, box, eps, dt=0.005, precision=precision, seed=9, step_engine=e,
                 self_mode=self_mode)
        g.init_field(x, q, m, v)
        out.append(g)
    return out


def same(a, b):
    for s, t in zip(a.fields() + a.particles(), b.fields() + b.particles()):
        assert np.array_equal(s, t)
    assert np.array_equal(a.forces(), b.forces())
    assert a.energy() == b.energy() and a.energy()["gauss_exact"] == 1.0


@pytest.mark.parametrize("mesh,n,cell", [((2, 3, 2), 2, 1.0), ((8, 8, 8), 16, 1.0),
                                         ((33, 9, 7), 130, 0.9), ((45, 38, 21), 600, 1.0),
                                         ((64, 40, 40), 4864, 1.0), ((30, 28, 26), 4866, 0.9),
                                         ((40, 40, 40), 9730, 1.0)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_single_launch_matches_graph(mesh, n, cell, precision):
    a, b = pair(mesh, n, precision, cell)
    for steps, th in ((1, TH), (2, TH), (35, TH), (4, None)):
        a.step(steps, th)
        b.step(steps, th)
        assert a.kernel_stats().single and not b.kernel_stats().single
    same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("n", [2, 600, 4866, 8194])
def test_host_loop_round_trip_matches_graph(n):
    a, b = pair((24, 20, 40), n, "fp32", 1.0, self_mode=2)
    for g in (a, b):
        io = g.io_buffers()
        x, v, img = g.particles()
        io["pos"][...], io["vel"][...], io["img"][...] = x, v, img
    for k in range(5):
        for g in (a, b):
            g.io_buffers()["vel"][...] *= 1.0 - 0.01 * k
            g.step_io(1, TH)
        for key in ("pos", "vel", "img", "f"):
            assert np.array_equal(a.io_buffers()[key], b.io_buffers()[key])
    a.step_io(7, TH, load=False)
    b.step_io(7, TH, load=False)
    assert np.array_equal(a.io_buffers()["f"], b.io_buffers()["f"])
    same(a, b)
    a.close()
    b.close()
