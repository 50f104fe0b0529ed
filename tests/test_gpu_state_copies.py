"""Host copies of a state: the packed blocks of a saved state, the fields and
the ledger against each other, word for word, on meshes and charge counts
that leave partial blocks (and none), in both precisions; and the energies'
background after a state with other valences was loaded."""
import numpy as np
import pytest

from paper_1309_7859_gb300 import inputs
from paper_1309_7859_gb300.inputs import EpsSpec

pytestmark = pytest.mark.gpu

HEADER = 96   # bytes before D in a saved state


def system(mesh, n, precision, seed):
    from paper_1309_7859_gb300.memd import Memd
    rng = np.random.default_rng(seed)
    box = tuple(float(N) for N in mesh)
    g = Memd(mesh, box, EpsSpec("const", 0, (2.0,)), dt=0.005, precision=precision, seed=seed)
    x = inputs.uniform_positions(rng, n, box)
    q = inputs.neutral_charges(rng, n)
    g.init_field(x, q, rng.uniform(0.5, 2.0, n), inputs.thermal_velocities(rng, n))
    g.step(3, (1.0, 1.0))
    return g


@pytest.mark.parametrize("mesh,n", [((3, 5, 7), 2), ((8, 8, 8), 0), ((33, 9, 7), 130),
                                    ((16, 16, 17), 256)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_saved_state_holds_the_fields_and_particles(mesh, n, precision):
    g = system(mesh, n, precision, 3)
    buf = g.save_state()
    V3 = 3 * g.V
    t = np.float32 if precision == "fp32" else np.float64
    D, B, Lg = g.fields()
    x, v, img = g.particles()
    at = HEADER
    for a in (D, B):
        assert np.array_equal(np.frombuffer(buf, t, V3, at), a.ravel().astype(t))
        at += V3 * t().itemsize
    assert np.array_equal(np.frombuffer(buf, np.int64, V3, at), Lg.ravel())
    at += 8 * V3
    for a in (x, v, g.forces()):
        assert np.array_equal(np.frombuffer(buf, np.float64, 3 * n, at), a.ravel())
        at += 24 * n
    assert np.array_equal(np.frombuffer(buf, np.int32, 3 * n, at + 24 * n), img.ravel())
    # into another system, and the ledger through set_fields
    h = system(mesh, n, precision, 4)
    h.load_state(buf)
    assert np.array_equal(h.save_state(), buf)
    h.set_fields(D=D, B=B, Lg=Lg)
    assert np.array_equal(h.save_state(), buf)
    eg, eh = g.energy(), h.energy()
    assert eg == eh and eh["gauss_exact"] == 1.0
    g.step(4)   # no thermostat: the two systems have noise keys of their own
    h.step(4)
    assert np.array_equal(g.save_state(), h.save_state())
    g.close()
    h.close()


def test_energy_background_follows_a_loaded_state():
    # 3 e over 512 vertices (a whole background), into a neutral system
    a = system((8, 8, 8), 2, "fp64", 5)
    b = system((8, 8, 8), 2, "fp64", 6)
    rng = np.random.default_rng(5)
    a.init_field(inputs.uniform_positions(rng, 2, (8.0,) * 3), np.array([1, 2], np.int32))
    b.load_state(a.save_state())
    ea, eb = a.energy(), b.energy()
    assert ea == eb and eb["gauss_exact"] == 1.0
    a.close()
    b.close()
