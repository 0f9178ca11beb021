"""The read-out of the bordered map at line lengths around its tiles (32 lanes, 4 elements
each, the short-line kernel below 24), against the allocation-free run, which accumulates
into an unpadded map and has no read-out: same photons, so the FP64 sums differ only by the
order of at most 2e4 additions per voxel; the conversions and the normalisation are exact
restatements in numpy."""
import numpy as np
import pytest

import workloads
from gpu_common import f32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    from paper_1711_03244_gb300 import build
    build.build()
    import paper_1711_03244_gb300 as m
    m.load()
    return m


@pytest.mark.parametrize("nx", [1, 5, 23, 24, 31, 33, 127, 128, 129, 161])
@pytest.mark.parametrize("gates", [1, 3, 70])
def test_readout_matches_unpadded_map(g, nx, gates):
    import torch
    ny, nz = 5, 7
    labels = np.ones((nz, ny, nx), dtype=np.uint8)
    labels[nz // 2:, ::2] = 2
    media = np.array([workloads.AIR, (0.02, 8.0, 0.9, 1.37), (0.1, 3.0, 0.5, 1.37)])
    wl = f32(workloads.c1(n_photons=20000).with_(labels=labels, media=media, src_pos=(nx / 2, 2.5, 0.0),
                                                 n_gates=gates, dt_ns=0.05))
    lab = torch.from_numpy(labels).cuda()
    flu = torch.empty((gates, nz, ny, nx), device="cuda", dtype=torch.float64)
    tally = torch.empty(g.NOALLOC_NOUT, device="cuda", dtype=torch.float64)
    cfg = g.mcx_run_cfg_default(n_photons=20000, n_gates=gates, dt_ns=wl.dt_ns, seed=4)
    g.mcx_run_noalloc(lab, wl.voxel_mm, wl.media, wl.src_kind, wl.src_pos, wl.src_dir, 0.0, cfg, flu, tally)
    torch.cuda.synchronize()
    ref = flu.cpu().numpy()
    eps = 20000 * 2.0 ** -53
    with g.Simulation.from_workload(wl) as sim:
        sim.run(20000, n_gates=gates, dt_ns=wl.dt_ns, seed=4)
        m64 = sim.fluence64()
        assert np.allclose(m64, ref, rtol=eps, atol=0)
        assert np.array_equal(sim.fluence(), m64.astype(np.float32))
        inv = np.zeros(3, dtype=np.float32)
        h = float(np.float32(wl.voxel_mm))
        for k in (1, 2):
            inv[k] = 1.0 / (float(np.float32(media[k, 0])) * h ** 3 * 20000.0 * float(np.float32(wl.dt_ns)))
        assert np.array_equal(sim.fluence64(normalized=True), m64 * inv.astype(np.float64)[labels])
        dev = torch.empty((gates, nz, ny, nx), device="cuda")
        sim.fluence(normalized=True, out=dev)
        assert np.array_equal(dev.cpu().numpy(), (m64 * inv.astype(np.float64)[labels]).astype(np.float32))
        sim.run(20000, n_gates=gates, dt_ns=wl.dt_ns, seed=4, accum_mode=0)
        assert np.allclose(sim.fluence(), ref, rtol=1e-3, atol=1e-6)
    with g.Batch() as b:
        b.add_workload(wl, n_photons=20000, seed=4)
        b.run(n_gates=gates, dt_ns=wl.dt_ns)
        fb = b.fluence(0)
        assert fb.sum(dtype=np.float64) == pytest.approx(ref.sum(), rel=1e-2)
        assert fb.shape == ref.shape and np.isfinite(fb).all()
