"""The row kernel's aligned cut (one mesh whose fields leave L2: every tile cut
at the same planes) against the halo-loop kernel, bit for bit, where tiles,
rows and planes do not divide evenly, for each width the kernel has."""
import numpy as np
import pytest

from paper_1309_7859_gb300 import inputs
from paper_1309_7859_gb300.inputs import EpsSpec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh,precision", [((256, 141, 83), "fp32"), ((132, 163, 131), "fp32"),
                                            ((128, 151, 71), "fp64")])
def test_aligned_rows_match_halo_loop(mesh, precision):
    from paper_1309_7859_gb300.memd import Memd
    rng = np.random.default_rng(mesh[1])
    box = tuple(float(N) for N in mesh)
    eps = EpsSpec("tanh", 1, (41.0, 39.0, 60.0, 20.0, 1.5))
    n = 20000
    x, q = inputs.uniform_positions(rng, n, box), inputs.neutral_charges(rng, n)
    v = inputs.thermal_velocities(rng, n)
    ref = None
    for kernel, shape in (("ldg", None), ("rows", (0, 0, 0, 256)), ("rows", (0, 0, 0, 512)),
                          ("auto", None)):
        g = Memd(mesh, box, eps, dt=0.005, precision=precision, field_kernel=kernel,
                 field_shape=shape, step_engine="graph")
        g.init_field(x, q, None, v)
        g.step(3)
        if kernel != "ldg":
            assert g.kernel_stats().field_kernel.startswith("k_rows")
        D, B, Lg = g.fields()
        if ref is None:
            ref = (D, B, Lg)
        for a, b in zip((D, B, Lg), ref):
            assert np.array_equal(a, b)
        g.close()
