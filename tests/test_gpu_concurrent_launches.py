"""Cooperative launches of several contexts at once, each on its own stream and
host thread: setups (the multigrid solve), single-launch steps, and steps of the
graph engine.  Each gives the bits it gives alone, and no bounded wait runs
out (a context would report it)."""
import threading

import numpy as np
import pytest

from paper_1309_7859_gb300 import inputs
from paper_1309_7859_gb300.inputs import EpsSpec

pytestmark = pytest.mark.gpu

TH = (1.0, 1.0)
# mesh, charges, precision, engine, steps a call, calls
JOBS = [((24, 20, 26), 300, "fp64", "single", 40, 6), ((32, 32, 32), 1000, "fp32", "single", 64, 8),
        ((30, 31, 33), 400, "fp64", "graph", 17, 4), ((16, 16, 16), 120, "fp32", "single", 1, 40),
        ((48, 40, 44), 900, "fp32", "auto", 9, 5)]


def work(job):
    from paper_1309_7859_gb300.memd import Memd
    mesh, n, precision, engine, k, calls = job
    out = []
    for seed in range(3):
        rng = np.random.default_rng(seed)
        box = tuple(float(N) for N in mesh)
        eps = EpsSpec("vertices", 0, (), inputs.smooth_random_vertices(rng, mesh, 1.0))
        x, q = inputs.uniform_positions(rng, n, box), inputs.neutral_charges(rng, n)
        g = Memd(mesh, box, eps, dt=0.005, precision=precision, seed=seed, step_engine=engine,
                 field_kernel="ldg", use_torch=False)
        g.init_field(x, q, None, inputs.thermal_velocities(rng, n))
        for _ in range(calls):
            g.step(k, TH)
        out.append(g.fields() + g.particles() + (g.forces(),))
        g.close()
    return out


def test_contexts_on_their_own_threads_match_alone():
    alone = [work(j) for j in JOBS]
    got, failed = [None] * len(JOBS), []

    def run(i):
        try:
            got[i] = work(JOBS[i])
        except Exception as e:      # a MemdError: reported below
            failed.append((JOBS[i], e))

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(JOBS))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    for a, b in zip(alone, got):
        for s, t in zip(a, b):
            assert all(np.array_equal(u, v) for u, v in zip(s, t))
