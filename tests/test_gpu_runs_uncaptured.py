"""Steps without graphs, which are launched in the runs that the graph engine
records, against the graph engine's steps one by one, bit for bit: single steps,
runs of every parity, a run and its remainder, row and tile kernels, few and
many charges and none."""
import numpy as np
import pytest

from paper_1309_7859_gb300 import inputs
from paper_1309_7859_gb300.inputs import EpsSpec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh,n,kernel", [((64, 24, 20), 900, "rows"), ((64, 24, 20), 900, "site"),
                                           ((24, 20, 40), 16390, "rows"), ((33, 18, 14), 0, "auto"),
                                           ((33, 18, 34), 16390, "ldg")])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_steps_without_graphs_match_single_steps(mesh, n, kernel, precision):
    from paper_1309_7859_gb300.memd import Memd
    rng = np.random.default_rng(n + mesh[0])
    box = tuple(float(N) for N in mesh)
    eps = EpsSpec("vertices", 0, (), inputs.smooth_random_vertices(rng, mesh, 1.0))
    x, q = inputs.uniform_positions(rng, n, box), inputs.neutral_charges(rng, n)
    v = inputs.thermal_velocities(rng, n)
    a, b = (Memd(mesh, box, eps, dt=0.005, precision=precision, seed=9, step_engine="graph",
                 field_kernel=kernel, use_graphs=g) for g in (False, True))
    for g in (a, b):
        g.init_field(x, q, None, v)
    for k in (1, 2, 5, 16, 19, 3):
        a.step(k, (1.0, 1.0))
        for _ in range(k):
            b.step(1, (1.0, 1.0))
    for s, t in zip(a.fields() + a.particles(), b.fields() + b.particles()):
        assert np.array_equal(s, t)
    assert np.array_equal(a.forces(), b.forces()) and a.energy() == b.energy()
    a.close()
    b.close()
