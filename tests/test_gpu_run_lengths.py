"""Recorded runs of steps of every kind of length (a length is recorded the third
time it is asked for with the same thermostat, up to 16 steps a run): short,
odd (the run ends on the other buffer), the longest, and one with a remainder,
each replayed from both buffer parities, against the same steps asked for one by
one, bit for bit.  Single systems with the row and the tile kernels, few and
many charges, sparse and dense application; batches likewise, one member without
charges."""
import numpy as np
import pytest

from paper_1309_7859_gb300 import inputs
from paper_1309_7859_gb300.inputs import EpsSpec

pytestmark = pytest.mark.gpu

TH = (1.0, 1.0)
# five calls a length: the third records it; odd lengths turn the parity at
# each call, single steps do it between the even ones
CALLS = [k for n in (2, 3, 5, 9, 15, 16, 19) for k in ([n] * 5 + [1] + [n] * 2)]


def make(mesh, n, precision, **kw):
    from paper_1309_7859_gb300.memd import Memd
    rng = np.random.default_rng(n + mesh[0])
    box = tuple(float(N) for N in mesh)
    eps = EpsSpec("vertices", 0, (), inputs.smooth_random_vertices(rng, mesh, 1.0))
    x, q = inputs.uniform_positions(rng, n, box), inputs.neutral_charges(rng, n)
    m, v = rng.uniform(0.5, 2.0, n), inputs.thermal_velocities(rng, n)
    g = Memd(mesh, box, eps, dt=0.005, precision=precision, seed=9, step_engine="graph", **kw)
    g.init_field(x, q, m, v)
    return g


def same(a, b):
    for s, t in zip(a.fields() + a.particles(), b.fields() + b.particles()):
        assert np.array_equal(s, t)
    assert np.array_equal(a.forces(), b.forces())
    assert a.energy() == b.energy() and a.energy()["gauss_exact"] == 1.0


def steps(a, b):
    for k in CALLS:
        a.step(k, TH)
        for _ in range(k):
            b.step(1, TH)


@pytest.mark.parametrize("mesh,n,kernel", [((40, 12, 10), 300, "rows"), ((17, 12, 9), 300, "site"),
                                           ((24, 20, 36), 16390, "rows"), ((25, 20, 36), 16390, "ldg")])
@pytest.mark.parametrize("precision,apply_mode", [("fp32", "sparse"), ("fp32", "dense"),
                                                  ("fp64", "sparse"), ("fp64", "dense")])
def test_recorded_lengths_match_single_steps(mesh, n, kernel, precision, apply_mode):
    a, b = (make(mesh, n, precision, field_kernel=kernel, apply_mode=apply_mode) for _ in range(2))
    steps(a, b)
    same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("meshes", [((8, 8, 8), (20, 16, 12), (16, 12, 20)),
                                    ((9, 8, 8), (20, 16, 12), (17, 12, 21))])
@pytest.mark.parametrize("counts", [(2, 0, 300), (0, 16390, 60)])
@pytest.mark.parametrize("precision,apply_mode", [("fp32", "sparse"), ("fp32", "dense"),
                                                  ("fp64", "sparse"), ("fp64", "dense")])
def test_batch_recorded_lengths_match_single_steps(meshes, counts, precision, apply_mode):
    import torch
    from paper_1309_7859_gb300.memd import Batch
    stream = torch.cuda.Stream()
    A, B = ([make(m, n, precision, stream=stream, apply_mode=apply_mode)
             for m, n in zip(meshes, counts)] for _ in range(2))
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
