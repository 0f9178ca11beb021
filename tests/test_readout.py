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


# an absorbing column (1 mean absorption length per voxel, no roulette): its map falls from
# about 2^13 to 2^-115, and the voxel size and the gate width take the normalisation's factor
# from 2^63 to 2^-81, so that products reach both far beyond 1 and below FP32's normal range,
# from factors of all sizes.  The FP32 read-out is the FP64 one rounded once more, bit for bit
# where the result is a normal number; below, the conversion may flush it.
@pytest.mark.parametrize("nx", [7, 33])
@pytest.mark.parametrize("h,dt", [(1e-12, 5.0), (1.0, 5.0), (1.0, 1e8), (1.0, 1e12), (1.0, 1e15), (1e5, 1e10)])
def test_readout_scales(g, nx, h, dt):
    import torch
    ny, nz, n = 5, 80, 20000
    labels = np.ones((nz, ny, nx), dtype=np.uint8)
    labels[:, :, ::2] = 2
    media = np.array([workloads.AIR, (1.0 / h, 0.05 / h, 0.8, 1.37), (1.01 / h, 0.04 / h, 0.8, 1.37)])
    wl = f32(workloads.c1(n_photons=n).with_(labels=labels, media=media, voxel_mm=h, src_kind=1, waist_mm=2 * h,
                                             src_pos=(nx * h / 2, 2.5 * h, 0.0), dt_ns=dt))
    tiny = 2.0 ** -126

    def check(got, m64):
        want = m64.astype(np.float32)
        normal = np.abs(want) >= tiny
        assert np.array_equal(got[normal], want[normal])
        assert (np.abs(got[~normal]) <= tiny).all()
        return normal & (want > 0)

    with g.Simulation.from_workload(wl) as sim:
        sim.run(n, dt_ns=wl.dt_ns, seed=4, rr_threshold=0.0, reflect=0)
        plain, norm = sim.fluence64(), sim.fluence64(normalized=True)
        assert check(sim.fluence(), plain).sum() > 400
        dev = torch.empty((1, nz, ny, nx), device="cuda")
        sim.fluence(normalized=True, out=dev)
        compared = check(dev.cpu().numpy(), norm)
        print(f"products from 2^{np.log2(norm[compared].min()):.0f} to 2^{np.log2(norm[compared].max()):.0f}")
        assert compared.sum() > 100


# the batch's read-out, element by element: against the single run's map (the same photons,
# as in the batch tests), and its normalisation against its own plain map, from which it
# differs by the two maps' roundings (FP32 sums are normalised in FP64 and rounded once)
@pytest.mark.parametrize("accum", [2, 0])
@pytest.mark.parametrize("nx", [5, 23, 24, 33, 129])
def test_batch_readout(g, nx, accum):
    ny, nz, gates, n = 5, 7, 3, 20000
    labels = np.ones((nz, ny, nx), dtype=np.uint8)
    labels[nz // 2:, ::2] = 2
    media = np.array([workloads.AIR, (0.02, 8.0, 0.9, 1.37), (0.1, 3.0, 0.5, 1.37)])
    wl = f32(workloads.c1(n_photons=n).with_(labels=labels, media=media, src_pos=(nx / 2, 2.5, 0.0)))
    with g.Simulation.from_workload(wl) as sim:
        sim.run(n, n_gates=gates, dt_ns=0.05, seed=4)
        ref = sim.fluence64()
    with g.Batch() as b:
        b.add_workload(wl, n_photons=10, seed=3)             # the second map starts elsewhere
        k = b.add_workload(wl, n_photons=n, seed=4)
        b.run(n_gates=gates, dt_ns=0.05, accum_mode=accum)
        plain, norm = b.fluence(k).astype(np.float64), b.fluence(k, normalized=True)
    assert np.linalg.norm(plain - ref) < 1e-3 * np.linalg.norm(ref)
    inv = np.zeros(3, dtype=np.float32)
    for m in (1, 2):
        inv[m] = 1.0 / (float(np.float32(media[m, 0])) * n * float(np.float32(0.05)))
    want = plain * inv.astype(np.float64)[labels]
    assert np.allclose(norm, want, rtol=2.0 ** (-22 if accum == 2 else -23), atol=0)


# widths on both sides of the rule (3/4 of a warp's lanes), maps on both sides of the short-line
# kernel's two forms, and line counts around its tiles, against the same photons in an unpadded map
@pytest.mark.parametrize("nx,ny,nz,gates", [(1, 1, 1, 1), (3, 1, 2, 1), (48, 9, 7, 3), (49, 9, 7, 3), (65, 64, 3, 2),
                                            (72, 64, 61, 5), (73, 5, 3, 2), (33, 193, 200, 1), (24, 128, 73, 66)])
def test_readout_kernels(g, nx, ny, nz, gates):
    import torch
    labels = np.ones((nz, ny, nx), dtype=np.uint8)
    labels[:, :, ::2] = 2
    media = np.array([workloads.AIR, (0.02, 8.0, 0.9, 1.37), (0.1, 3.0, 0.5, 1.37)])
    wl = f32(workloads.c1(n_photons=20000).with_(labels=labels, media=media, src_kind=1, waist_mm=max(2.0, ny / 4),
                                                 src_pos=(nx / 2, ny / 2, 0.0)))
    with g.Simulation.from_workload(wl) as sim:
        sim.run(20000, n_gates=gates, dt_ns=0.02, seed=4)
        plain = sim.fluence64()
        assert plain.sum() > 0
        inv = np.zeros(3, dtype=np.float32)
        for k in (1, 2):
            inv[k] = 1.0 / (float(np.float32(media[k, 0])) * 20000.0 * float(np.float32(0.02)))
        want = plain * inv.astype(np.float64)[labels]
        for normalized, m64 in ((False, plain), (True, want)):
            assert np.array_equal(sim.fluence64(normalized=normalized), m64)
            dev = torch.empty((gates, nz, ny, nx), device="cuda")
            sim.fluence(normalized=normalized, out=dev)
            assert np.array_equal(dev.cpu().numpy(), m64.astype(np.float32))
        total = sim.tally()["absorbed"]
    assert plain.sum() == pytest.approx(total, rel=1e-5)
    # the same photons into an unpadded map, which is read as it is
    lab = torch.from_numpy(labels).cuda()
    flu = torch.empty((gates, nz, ny, nx), device="cuda", dtype=torch.float64)
    tally = torch.empty(g.NOALLOC_NOUT, device="cuda", dtype=torch.float64)
    cfg = g.mcx_run_cfg_default(n_photons=20000, n_gates=gates, dt_ns=0.02, seed=4)
    g.mcx_run_noalloc(lab, wl.voxel_mm, wl.media, wl.src_kind, wl.src_pos, wl.src_dir, wl.waist_mm, cfg, flu, tally)
    torch.cuda.synchronize()
    assert np.allclose(plain, flu.cpu().numpy(), rtol=20000 * 2.0 ** -53, atol=0)
