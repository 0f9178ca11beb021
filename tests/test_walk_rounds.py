"""The walk's rounds: how a short run's photons are shared out among lanes, and the rarely
taken path of a segment (gate changes, the time limit, the event cap, the roulette,
near-axial directions), where each can go wrong.

A run is a function of (seed, photon ids), so the sharing must not change a single photon:
those comparisons are exact.  The rare path runs in the FP64 instantiation against the
oracle: both follow the same decisions, up to photons whose FP64 rounding meets one of
them (at most 1 in 1000, as in the other fixed-seed tests).
"""
import numpy as np
import pytest

import workloads
from gpu_common import F32_RR, balance, f32, gpu_run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    from paper_1711_03244_gb300 import build
    build.build()
    import paper_1711_03244_gb300 as m
    m.load()
    return m


@pytest.fixture(scope="module")
def reference(g):
    """600 photons with every lane of the default grid open to the first claims"""
    return gpu_run(f32(workloads.c1()), n_photons=600, exit_log=600, seed=5)


# 4 blocks of 64 threads: 8 warps, 256 lanes; a block's share fills one warp at 128 photons
@pytest.mark.parametrize("n", [1, 3, 4, 5, 127, 128, 129, 255, 256, 257, 600])
@pytest.mark.parametrize("block,grid", [(64, 4), (32, 1), (256, 0)])
def test_sharing_does_not_change_photons(g, reference, n, block, grid):
    r = gpu_run(f32(workloads.c1()), n_photons=n, exit_log=600, seed=5, block_size=block, grid_size=grid)
    assert r["stats"]["photons"] == n
    assert np.array_equal(r["exits"][:n], reference["exits"][:n])
    assert balance(r["tally"]) == pytest.approx(n, rel=1e-6)


# photon counts at which the grid changes (2.6, 3.5, 13 and 26 photons per lane of 4, 8, 16
# and 24 warps on each of 152 SMs), each against the full grid
@pytest.mark.parametrize("n", [50585, 50586, 136192, 136193, 1011712, 1011713, 3035136, 3035137])
@pytest.mark.parametrize("block", [0, 128])
def test_grid_by_photon_count(g, n, block):
    wl = f32(workloads.c1(n_photons=n).with_(labels=np.ones((8, 8, 8), dtype=np.uint8), src_pos=(4.0, 4.0, 0.0)))
    a = gpu_run(wl, exit_log=n, seed=9, block_size=block)
    b = gpu_run(wl, exit_log=n, seed=9, block_size=block, grid_size=152 * (4 if block == 0 else 8))
    assert a["stats"] == b["stats"] and a["stats"]["photons"] == n
    assert np.array_equal(a["exits"], b["exits"])
    assert np.allclose(a["energy"], b["energy"], rtol=1e-6)


@pytest.mark.parametrize("case", ["gates", "limit", "cap", "roulette", "axial"])
def test_rare_path_matches_oracle(g, case):
    import oracle as orc
    n, kw, okw = 1000, {}, {}
    wl = f32(workloads.c1(n_photons=n).with_(labels=np.ones((16, 16, 16), dtype=np.uint8),
                                             src_pos=(8.0, 8.0, 0.0)))
    if case == "gates":                       # gates as long as a mean free path
        wl = f32(wl.with_(n_gates=200, dt_ns=0.0005))
    elif case == "limit":                     # most photons end at the limit
        wl = f32(wl.with_(n_gates=3, dt_ns=0.02))
    elif case == "cap":
        kw["max_events"] = okw["max_events"] = 257
    elif case == "roulette":
        kw["rr_threshold"] = okw["rr_threshold"] = float(np.float32(0.7))
        kw["rr_m"] = okw["rr_m"] = 2.0
    else:                                     # forward scattering within 0.5 degrees of the axis
        wl = f32(wl.with_(media=np.array([workloads.AIR, (0.01, 1.0, 0.9999, 1.37)])))
    g64 = gpu_run(wl, exit_log=n, precision=1, **{"rr_threshold": F32_RR, **kw})
    o = orc.run(wl, exit_cap=n, **{"rr_threshold": F32_RR, **okw})
    same = (g64["exits"]["fate"] == o.exits["fate"]) & (g64["exits"]["nscat"] == o.exits["nscat"])
    print(f"{case}: {same.mean():.4f} of the photons match")
    assert same.mean() >= 0.999
    # a deposit moves to the neighbouring gate where the two roundings of a time meet its
    # edge: at most one photon's weight in 1000
    d = np.abs(g64["energy"].astype(np.float64).reshape(-1) - o.energy.reshape(-1)).sum()
    assert d <= 2e-3 * o.energy.sum()


# beams whose first voxels are summed per warp, against the same run with every deposit sent
# to the map (an unused medium that scatters strongly turns the sums off): the FP64 sums are
# regrouped, so they agree to FP64 rounding over 2e4 additions
@pytest.mark.parametrize("block", [32, 256])
@pytest.mark.parametrize("name,pos,direction,reflect,gates", [
    ("z", (30.0, 30.0, 0.0), (0.0, 0.0, 1.0), 0, 1),
    ("z_reflect_gates", (30.0, 30.0, 0.0), (0.0, 0.0, 1.0), 1, 7),
    ("inside_down", (10.5, 20.25, 33.75), (0.0, 0.0, -1.0), 1, 1),
    ("x_from_far_face", (60.0, 12.0, 7.5), (-1.0, 0.0, 0.0), 1, 2),
    ("oblique", (0.0, 17.3, 4.2), (0.6, 0.64, 0.48), 1, 1),
    ("corner", (0.0, 0.0, 0.0), (1.0, 1.0, 1.0), 1, 1),
    ("last_voxel", (59.5, 59.5, 59.5), (0.0, 0.0, 1.0), 1, 1),
])
@pytest.mark.parametrize("variant", ["B1", "B2A"])
def test_beam_voxel_sums(g, variant, name, pos, direction, reflect, gates, block):
    wl = f32(workloads.paper_b(variant, n_photons=20000).with_(src_pos=pos, src_dir=direction))
    maps, stats = [], []
    for media in (wl.media, np.concatenate([wl.media, [[0.01, 100.0, 0.9, 1.37]]])):
        with g.Simulation.from_workload(wl.with_(media=media)) as sim:
            sim.run(20000, n_gates=gates, dt_ns=0.2, seed=3, reflect=reflect, block_size=block)
            maps.append(sim.fluence64())
            stats.append(sim.stats())
    assert stats[0] == stats[1]
    assert np.array_equal(maps[0] > 0, maps[1] > 0)
    assert np.allclose(maps[0], maps[1], rtol=20000 * 2.0 ** -53, atol=0)


# the same sums in the allocation-free run, whose map has no border, on an odd-sized volume, and
# in a run with detectors, each against its run with every deposit sent to the map
@pytest.mark.parametrize("pos,direction", [((20.0, 8.0, 0.0), (0.0, 0.0, 1.0)), ((0.0, 5.5, 3.25), (1.0, 0.0, 0.0)),
                                           ((41.0, 17.0, 23.0), (-0.6, -0.64, -0.48)), ((40.5, 16.5, 22.5), (0.0, 1.0, 0.0))])
@pytest.mark.parametrize("gates", [1, 3])
def test_beam_voxel_sums_unpadded(g, pos, direction, gates):
    import torch
    labels = np.ones((23, 17, 41), dtype=np.uint8)
    labels[5:9, 4:12, 10:30] = 2
    media = np.array([workloads.AIR, (0.01, 1.0, 0.1, 1.37), (0.02, 5.0, 0.8, 1.2)])
    lab = torch.from_numpy(labels).cuda()
    maps, tallies = [], []
    for m in (media, np.concatenate([media, [[0.01, 100.0, 0.9, 1.37]]])):
        flu = torch.empty((gates,) + labels.shape, device="cuda", dtype=torch.float64)
        tally = torch.zeros(g.NOALLOC_NOUT, device="cuda", dtype=torch.float64)
        cfg = g.mcx_run_cfg_default(n_photons=20000, n_gates=gates, dt_ns=0.1, seed=3)
        g.mcx_run_noalloc(lab, 1.0, m, 0, pos, direction, 0.0, cfg, flu, tally)
        torch.cuda.synchronize()
        maps.append(flu.cpu().numpy())
        tallies.append(tally.cpu().numpy())
    assert np.array_equal(maps[0] > 0, maps[1] > 0)
    assert np.allclose(maps[0], maps[1], rtol=20000 * 2.0 ** -53, atol=0)
    assert np.allclose(tallies[0], tallies[1], rtol=1e-12)
    wl = f32(workloads.c1(n_photons=20000).with_(labels=labels, media=media, src_pos=pos, src_dir=direction))
    with g.Simulation.from_workload(wl) as sim:
        sim.run(20000, n_gates=gates, dt_ns=0.1, seed=3)
        assert np.allclose(sim.fluence64(), maps[0], rtol=20000 * 2.0 ** -53, atol=0)


def test_beam_voxel_sums_with_detectors(g):
    wl = f32(workloads.paper_b("B2A", n_photons=20000))
    det = np.array([[30.0, 30.0, 60.0, 15.0], [20.0, 30.0, 0.0, 4.0]])
    maps, stats, records = [], [], []
    for media in (wl.media, np.concatenate([wl.media, [[0.01, 100.0, 0.9, 1.37]]])):
        with g.Simulation.from_workload(wl.with_(media=media, detectors=det)) as sim:
            sim.run(20000, n_gates=2, dt_ns=0.2, seed=3, max_detected=20000)
            maps.append(sim.fluence64())
            stats.append(sim.stats())
            records.append(sim.detected())
    assert stats[0] == stats[1] and stats[0]["detected"] > 100
    assert np.allclose(maps[0], maps[1], rtol=20000 * 2.0 ** -53, atol=0)
    (a, n), (b, m) = records
    assert n == m
    for k in a:                               # the unused medium adds a column of partial paths
        assert np.array_equal(a[k], b[k][..., :a[k].shape[1]] if k == "ppath" else b[k]), k


# the same on both sides of the other limits: a map past L2 (8^3 voxels in 40 000 gates), a short
# window, the compensated mode, a medium that hardly scatters, the FP64 walk; the counts lie
# beside the limits of 8, 16 and 24 warps per SM of 152 (FP64: 4)
GRIDS = {
    "large map": (dict(gates=40_000, dt=5 / 40_000), [136192, 136193, 505856, 505857, 1517568, 1517569]),
    "window": (dict(gates=1, dt=0.3), [13619, 13620, 101171, 101172, 303513, 303514]),
    "compensated": (dict(accum=1), [20_000, 60_000, 250_000, 600_000, 1_600_000]),
    "clear": (dict(mus=0.1), [34048, 34049, 252928, 252929, 758784, 758785]),
    "fp64": (dict(precision=1), [20_000, 50585, 50586]),
}


@pytest.mark.parametrize("case,n", [(c, n) for c in GRIDS for n in GRIDS[c][1]])
def test_grid_does_not_change_photons(g, case, n):
    kw = GRIDS[case][0]
    gates, dt = kw.get("gates", 1), kw.get("dt", 5.0)
    media = np.array([workloads.AIR, (0.01, kw.get("mus", 10.0), 0.9, 1.37)])
    wl = f32(workloads.c1(n_photons=n).with_(labels=np.ones((8, 8, 8), dtype=np.uint8), media=media,
                                             src_pos=(4.0, 4.0, 0.0), n_gates=gates, dt_ns=dt))
    run = dict(exit_log=n, seed=9, accum_mode=kw.get("accum", 2), precision=kw.get("precision", 0))
    a = gpu_run(wl, **run)
    b = gpu_run(wl, grid_size=152 * 4, **run)
    assert a["stats"] == b["stats"] and a["stats"]["photons"] == n
    assert np.array_equal(a["exits"], b["exits"])
    assert np.allclose(a["energy"], b["energy"], rtol=1e-6)


@pytest.mark.parametrize("n", [389119, 389120, 389121, 1556480, 1556481, 3969024, 3969025])
def test_batch_grid_does_not_change_photons(g, n):
    wls = [f32(workloads.c1(n_photons=k).with_(labels=np.ones((16, 16, 16), dtype=np.uint8), src_pos=(8.0, 8.0, 0.0),
                                               n_gates=1, dt_ns=5.0, seed=k)) for k in (n // 3, n - n // 3)]
    res = []
    with g.Batch() as b:
        for wl in wls:
            b.add_workload(wl)
        for kw in ({}, {"grid_size": 152 * 4}):
            b.run(n_gates=1, dt_ns=5.0, **kw)
            res.append((b.stats(), [b.tally(i) for i in range(2)], [b.fluence(i) for i in range(2)]))
    assert res[0][0] == res[1][0] and res[0][0]["photons"] == n
    for i in range(2):
        for k in res[0][1][i]:
            assert res[0][1][i][k] == pytest.approx(res[1][1][i][k], rel=1e-11, abs=1e-11)
        assert np.allclose(res[0][2][i], res[1][2][i], rtol=1e-6)


def test_static_split_of_more_threads_than_32_bits_count(g):
    """The thread-level split over a grid whose threads just exceed 2^32: a thread takes at most
    one of the photons, and each photon once."""
    wl = f32(workloads.c1(n_photons=600).with_(labels=np.ones((8, 8, 8), dtype=np.uint8), src_pos=(4.0, 4.0, 0.0)))
    a = gpu_run(wl, exit_log=600, seed=5)
    b = gpu_run(wl, exit_log=600, seed=5, claim_mode=1, grid_size=2 ** 24)
    assert b["stats"] == a["stats"] and np.array_equal(a["exits"], b["exits"])
    assert balance(b["tally"]) == pytest.approx(600, rel=1e-6)
