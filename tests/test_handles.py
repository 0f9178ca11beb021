"""Several simulations alive at once: each keeps its launch shape, so a run must not depend on
which handle asked for one last."""
import numpy as np
import pytest

import workloads
from gpu_common import f32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("accum,precision", [(2, 0), (0, 0), (1, 0), (2, 1)])
def test_run_after_a_smaller_handle(accum, precision):
    from paper_1711_03244_gb300 import build
    build.build()
    import paper_1711_03244_gb300 as g
    g.load()
    wl = f32(workloads.c1(n_photons=500))
    many = np.concatenate([wl.media] + [wl.media[1:]] * 200)
    with g.Simulation.from_workload(wl.with_(media=many)) as a, g.Simulation.from_workload(wl) as b:
        kw = dict(seed=3, accum_mode=accum, precision=precision)
        a.run(500, **kw)
        first = a.fluence()
        b.run(500, **kw)
        a.run(500, **kw)
        assert np.array_equal(a.fluence() > 0, first > 0)
        assert np.allclose(a.fluence(), first, rtol=1e-5)
