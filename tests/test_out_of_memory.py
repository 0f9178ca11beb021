"""Calls that ask for more memory than the device has: they say so, and leave a handle that
works.  The sizes are far beyond any device's, so that the allocation itself is refused."""
import numpy as np
import pytest

import workloads
from gpu_common import f32

pytestmark = pytest.mark.gpu

GATES = 2 ** 31                       # 16 GiB of map per voxel


@pytest.fixture(scope="module")
def g():
    from paper_1711_03244_gb300 import build
    build.build()
    import paper_1711_03244_gb300 as m
    m.load()
    return m


def refused(g, call):
    with pytest.raises(g.McxError) as e:
        call()
    assert e.value.status == g.MCX_E_OOM


def test_next_call_after_a_refused_run(g):
    """The refusal is reported once, by the call that met it."""
    wl = f32(workloads.c1(n_photons=2000))
    with g.Simulation.from_workload(wl) as a, g.Simulation.from_workload(wl) as b, g.Batch() as c:
        c.add_workload(wl)
        refused(g, lambda: a.run(2000, n_gates=GATES, dt_ns=1e-9))
        b.run(2000, seed=3)
        refused(g, lambda: c.run(n_gates=GATES, dt_ns=1e-9))
        a.run(2000, seed=3)
        refused(g, lambda: c.run(n_gates=GATES, dt_ns=1e-9))
        c.run(n_gates=1, dt_ns=5.0)
        assert c.stats()["photons"] == 2000
        assert a.stats() == b.stats() and np.allclose(a.fluence(), b.fluence(), rtol=1e-6)
