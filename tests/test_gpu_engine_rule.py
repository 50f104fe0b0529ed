"""The engine that a host round trip of one step takes when left to choose: the
single launch up to 48^3 in both precisions, the graph beyond its limits; the
same results as with the graph asked for."""
import numpy as np
import pytest

from paper_1309_7859_gb300 import inputs
from paper_1309_7859_gb300.inputs import EpsSpec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,precision,single", [(48, "fp32", True), (48, "fp64", True),
                                                (51, "fp32", False), (49, "fp64", False)])
def test_round_trip_engine(N, precision, single):
    from paper_1309_7859_gb300.memd import Memd
    rng = np.random.default_rng(N)
    n, box = 500, (float(N),) * 3
    x, q = inputs.uniform_positions(rng, n, box), inputs.neutral_charges(rng, n)
    v = inputs.thermal_velocities(rng, n)
    out = []
    for engine in ("auto", "graph"):
        g = Memd((N, N, N), box, EpsSpec("const", 0, (3.0,)), dt=0.005, precision=precision,
                 step_engine=engine)
        g.init_field(x, q, None, v)
        io = g.io_buffers()
        for _ in range(3):
            io["pos"][...], io["vel"][...], io["img"][...] = g.particles()
            g.step_io(1, (1.0, 1.0), load=True)
            if engine == "auto":
                assert g.kernel_stats().single == single
        out.append(g.fields() + g.particles() + (g.forces(),))
        g.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
