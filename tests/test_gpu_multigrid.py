"""The multigrid solve of the effective permittivity and the initial field
at the sizes where its levels change: extents of 2 and 3, odd extents (three
colours, a seam), axes that reach one vertex before the others, and meshes
on either side of the largest level that one CTA takes (343 vertices), with
smooth profiles and a random permittivity on every link.  Against the FP64
oracle, whose relaxation is another method altogether: the tolerances are
those of the other initial-solution tests (two solvers stopped at a residual
of 1e-12 differ by up to the operator's condition number times it)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1309_7859_gb300 import inputs
from paper_1309_7859_gb300.inputs import EpsSpec

pytestmark = pytest.mark.gpu

MESHES = [(2, 2, 2), (3, 3, 3), (2, 5, 9), (7, 7, 7), (8, 7, 7), (3, 2, 60), (16, 12, 11),
          (17, 17, 17), (24, 20, 12)]


@pytest.mark.parametrize("mesh", MESHES)
@pytest.mark.parametrize("kind", ["vertices", "links"])
def test_eps_eff_and_initial_field_match_oracle(mesh, kind):
    from paper_1309_7859_gb300.memd import Memd
    rng = np.random.default_rng(sum(mesh))
    V = mesh[0] * mesh[1] * mesh[2]
    box = tuple(0.5 * N for N in mesh)
    if kind == "vertices":
        vals = inputs.smooth_random_vertices(rng, mesh, 1.0)
    else:
        vals = rng.uniform(2.0, 80.0, size=3 * V)
    eps = EpsSpec(kind, 0, (), vals)
    okind = {"vertices": O.EPS_VERTICES, "links": O.EPS_LINKS}[kind]
    n = 2 * max(1, min(40, V // 8))
    x, q = inputs.uniform_positions(rng, n, box), inputs.neutral_charges(rng, n)
    g = Memd(mesh, box, eps, c_light=1.0, dt=0.005, precision="fp64")
    o = O.OracleSystem(mesh, box, eps=dict(kind=okind, axis=0, params=(), values=vals),
                       c_light=1.0, dt=0.005)
    _, _, M = g.setup()
    assert np.max(np.abs(M - o.Minv)) < 1e-10 * np.max(np.abs(o.Minv))
    o.set_particles(x, q)
    o.init_field()
    g.init_field(x, q)
    D, _, Lg = g.fields()
    Do = o.field("D")
    assert np.array_equal(Lg, o.field("Lg"))
    assert np.sqrt(np.sum((D - Do) ** 2) / np.sum(Do ** 2)) < 1e-9
    g.close()
