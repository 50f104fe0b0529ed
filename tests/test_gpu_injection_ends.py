"""An injected barrier fault ends with the report of its timeout: a context left
to choose its engine then steps as it did before."""
import numpy as np
import pytest

from paper_1309_7859_gb300 import inputs
from paper_1309_7859_gb300.inputs import EpsSpec

pytestmark = pytest.mark.gpu


def test_engine_choice_returns_after_the_timeout():
    from paper_1309_7859_gb300.memd import Memd, MemdError
    mesh, n = (40, 36, 38), 400        # the graph, but for host round trips of one step
    rng = np.random.default_rng(2)
    box = tuple(float(N) for N in mesh)
    x, q = inputs.uniform_positions(rng, n, box), inputs.neutral_charges(rng, n)
    g, ref = (Memd(mesh, box, EpsSpec("const", 0, (2.0,)), dt=0.005, precision="fp32") for _ in range(2))
    for s in (g, ref):
        s.init_field(x, q)
        s.step(2)
    assert not g.kernel_stats().single
    saved = g.save_state()
    g.inject("barrier_skew", wait_s=0.002)
    g.step(1)
    assert g.kernel_stats().single
    with pytest.raises(MemdError) as err:
        g.energy()
    assert err.value.status == 9       # MEMD_ERR_TIMEOUT
    g.inject("none")
    g.load_state(saved)
    g.step(3)
    ref.step(3)
    assert not g.kernel_stats().single
    for a, b in zip(g.fields() + g.particles(), ref.fields() + ref.particles()):
        assert np.array_equal(a, b)
    g.close()
    ref.close()
