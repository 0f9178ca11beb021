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


def test_recorded_batch_after_a_refused_autotuning(g):
    """The autotuner's trials have written the maps and moved buffers that the recorded run
    points to, also when one of them is refused: the next run records anew, and there is no
    result to read until it has run."""
    wls = [f32(w).with_(n_photons=20_000) for w in workloads.c4(n_sims=3)]
    with g.Batch() as b:
        for wl in wls:
            b.add_workload(wl)
        b.run(n_gates=5, dt_ns=1.0, use_graph=1)
        first = [b.fluence(i) for i in range(len(wls))]
        refused(g, lambda: b.autotune(n_gates=GATES, dt_ns=1e-9))
        with pytest.raises(g.McxError) as e:
            b.stats()
        assert e.value.status == g.MCX_E_STATE
        b.run(n_gates=5, dt_ns=1.0, use_graph=1)
        assert b.stats()["photons"] == 60_000
        for i, m in enumerate(first):
            assert np.allclose(b.fluence(i), m, rtol=1e-6, atol=0)


def test_no_result_after_a_refused_run(g):
    """A run that is refused memory has given up the map of the one before: reading it is
    refused in turn, until a run succeeds.  Refused arguments leave the results alone."""
    wl = f32(workloads.c1(n_photons=2000))
    with g.Simulation.from_workload(wl) as a, g.Batch() as b:
        b.add_workload(wl)
        a.run(2000, seed=3)
        b.run(n_gates=1, dt_ns=5.0)
        before = a.fluence(), b.fluence(0)
        for bad in (lambda: a.run(2000, n_gates=0), lambda: b.run(n_gates=0)):
            with pytest.raises(g.McxError) as e:
                bad()
            assert e.value.status == g.MCX_E_ARG
        a.n_gates = b.n_gates = 1
        assert np.array_equal(a.fluence(), before[0]) and np.array_equal(b.fluence(0), before[1])
        for accum in (2, 0):
            refused(g, lambda: a.run(2000, n_gates=GATES, dt_ns=1e-9, accum_mode=accum))
            refused(g, lambda: b.run(n_gates=GATES, dt_ns=1e-9, accum_mode=accum))
            a.n_gates = b.n_gates = 1
            for read in (a.fluence, a.fluence64, a.tally, a.stats, lambda: b.fluence(0), lambda: b.tally(0), b.stats):
                with pytest.raises(g.McxError) as e:
                    read()
                assert e.value.status == g.MCX_E_STATE
            a.run(2000, seed=3)
            b.run(n_gates=1, dt_ns=5.0)
            assert np.allclose(a.fluence(), before[0], rtol=1e-6)
            assert np.allclose(b.fluence(0), before[1], rtol=1e-6)
