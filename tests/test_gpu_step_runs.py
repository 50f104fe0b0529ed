"""Steps of the graph engine asked for together, which it runs as graphs of
eight steps, against the same steps asked for one by one, bit for bit: both
buffer parities, remainders, a second thermostat, few and many charges, every
field kernel, alone and in a batch."""
import numpy as np
import pytest

from paper_1309_7859_gb300 import inputs
from paper_1309_7859_gb300.inputs import EpsSpec

pytestmark = pytest.mark.gpu

TH = (1.0, 1.0)


def make(mesh, n, precision, engine="graph", **kw):
    from paper_1309_7859_gb300.memd import Memd
    rng = np.random.default_rng(n + mesh[0])
    box = tuple(float(N) for N in mesh)
    eps = EpsSpec("vertices", 0, (), inputs.smooth_random_vertices(rng, mesh, 1.0))
    x, q = inputs.uniform_positions(rng, n, box), inputs.neutral_charges(rng, n)
    m, v = rng.uniform(0.5, 2.0, n), inputs.thermal_velocities(rng, n)
    g = Memd(mesh, box, eps, dt=0.005, precision=precision, seed=9, step_engine=engine, **kw)
    g.init_field(x, q, m, v)
    return g


def same(a, b):
    for s, t in zip(a.fields() + a.particles(), b.fields() + b.particles()):
        assert np.array_equal(s, t)
    assert np.array_equal(a.forces(), b.forces())
    assert a.energy() == b.energy() and a.energy()["gauss_exact"] == 1.0


def steps(a, b):
    """a together, b one by one: shorter than a run, a run from the odd
    parity with a remainder, two thermostats, none"""
    for n, th in ((3, TH), (41, TH), (32, TH), (35, (0.5, 2.0)), (64, None), (7, None)):
        a.step(n, th)
        for _ in range(n):
            b.step(1, th)


@pytest.mark.parametrize("mesh,n", [((4, 6, 5), 2), ((33, 18, 14), 600), ((24, 20, 40), 16390)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("apply_mode", ["sparse", "dense"])
def test_runs_match_single_steps(mesh, n, precision, apply_mode):
    a, b = (make(mesh, n, precision, apply_mode=apply_mode) for _ in range(2))
    steps(a, b)
    same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("kernel", ["ldg", "site", "tma", "rows"])
def test_runs_match_single_steps_of_every_field_kernel(kernel):
    a, b = (make((64, 24, 20), 900, "fp32", field_kernel=kernel) for _ in range(2))
    steps(a, b)
    same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("counts", [(2, 130, 600), (300, 16390, 60)])
def test_batch_runs_match_single_steps(counts, precision):
    import torch
    from paper_1309_7859_gb300.memd import Batch
    stream = torch.cuda.Stream()
    meshes = ((8, 8, 8), (20, 16, 24), (17, 12, 9))
    A, B = ([make(m, n, precision, stream=stream) for m, n in zip(meshes, counts)]
            for _ in range(2))
    a, b = Batch(A), Batch(B)
    steps(a, b)
    a.synchronize()
    b.synchronize()
    for s, t in zip(A, B):
        same(s, t)
    a.close()
    b.close()
    for g in A + B:
        g.close()


def test_engine_chosen_call_by_call_matches_graph():
    """a mesh that takes the single launch in host round trips, the graph
    otherwise"""
    a, b = (make((40, 36, 38), 1200, "fp32", engine=e) for e in ("auto", "graph"))
    seen = []
    for n in (20, 1, 3, 1, 20, 20, 1):
        for g in (a, b):
            if n == 1:
                io = g.io_buffers()
                io["pos"][...], io["vel"][...], io["img"][...] = g.particles()
                g.step_io(1, TH)
            else:
                g.step(n, TH)
        seen.append(a.kernel_stats().single)
    assert seen == [n == 1 for n in (20, 1, 3, 1, 20, 20, 1)]
    same(a, b)
    a.close()
    b.close()
