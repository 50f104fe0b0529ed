"""Every row-kernel width that the autotuner can choose can also be asked for:
576 threads a CTA, alone and in a batch, against the halo-loop kernel, bit for
bit, with FP32 and FP64 fields, on a mesh whose fields fit L2 (the balanced cut)
and on one whose fields do not (every tile cut at the same planes)."""
import numpy as np
import pytest

from paper_1309_7859_gb300 import inputs
from paper_1309_7859_gb300.inputs import EpsSpec

pytestmark = pytest.mark.gpu

WIDE = dict(field_kernel="rows", field_shape=(0, 0, 0, 576))


def make(mesh, precision, stream=None, **kw):
    from paper_1309_7859_gb300.memd import Memd
    rng = np.random.default_rng(mesh[1])
    box = tuple(float(N) for N in mesh)
    eps = EpsSpec("tanh", 1, (41.0, 39.0, 0.4 * box[1], box[1] / 7, 1.5))
    n = 600
    x, q = inputs.uniform_positions(rng, n, box), inputs.neutral_charges(rng, n)
    g = Memd(mesh, box, eps, dt=0.005, precision=precision, step_engine="graph", stream=stream, **kw)
    g.init_field(x, q, None, inputs.thermal_velocities(rng, n))
    return g


def same(a, b):
    for s, t in zip(a.fields() + a.particles(), b.fields() + b.particles()):
        assert np.array_equal(s, t)


@pytest.mark.parametrize("mesh,precision", [((64, 37, 21), "fp32"), ((256, 141, 83), "fp32"),
                                            ((4, 5, 6), "fp32"), ((36, 23, 30), "fp64"),
                                            ((128, 151, 71), "fp64")])
def test_width_576_matches_halo_loop(mesh, precision):
    a, b = make(mesh, precision, **WIDE), make(mesh, precision, field_kernel="ldg")
    a.step(3)
    b.step(3)
    assert a.kernel_stats().field_kernel == "k_rows<nt=576>"
    same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_members_fixing_width_576_fix_the_batch(precision):
    import torch
    from paper_1309_7859_gb300.memd import Batch
    stream = torch.cuda.Stream()
    meshes = ((8, 9, 10), (40, 16, 24), (64, 33, 21))
    A = [make(m, precision, stream, **WIDE) for m in meshes]
    B = [make(m, precision, field_kernel="ldg") for m in meshes]
    batch = Batch(A)
    batch.step(4)
    batch.synchronize()
    assert batch.kernel_stats().field_kernel == "k_rows_batch<nt=576>"
    for a, b in zip(A, B):
        b.step(4)
        same(a, b)
    batch.close()
    for g in A + B:
        g.close()
