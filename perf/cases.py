"""What the library's speed is measured on: one photon run, batch or network pass per case,
each through the calls that a program makes.

Walk cases run one simulation and read its results the way the drivers of the library do
(fluence map into a device tensor, energy tallies and detected records to the host).  The
problems are the workloads of this repository: the homogeneous cube, the two spheres with
disk detectors, the layered tissue, the paper's benchmarks B1 and B2a, and volumes of random
ellipsoids like the batched ones, at the sizes and photon counts that fit a short pass.
Denoiser cases run the network on maps of the 64 mm cubes it is trained on, and on a wider
volume with medium features.

A run is a function of (problem, seed, photon range) alone, so the same case and seed give
the same map.  `exact` gives the network's outputs in 64 bits; a photon walk has no such
value (a photon's path is decided by the 32-bit arithmetic of thousands of events in a row).
"""
import math

import numpy as np
import torch

import paper_1711_03244_gb300 as mcx
import workloads

GATES = {"cube": (1, 5.0), "spheres": (10, 0.5), "layers": (50, 0.1), "b1": (1, 5.0), "b2a": (1, 5.0)}
# arithmetic operations of one photon's history (segments, hops, scatterings, faces), the
# mean over each problem's photons; the random ellipsoids' mean is over many such volumes
OPS = {"cube": 1.59e5, "spheres": 1.42e5, "layers": 1.14e5, "b1": 1.5e4, "b2a": 2.7e4, "ellipsoids": 6e4}


def listed():
    return [
        # a first look at a problem: few photons, where launches, waits and the longest
        # single photon history count
        {"name": "walk_cube_2e4", "kind": "walk", "problem": "cube", "nx": 64, "ny": 64, "nz": 64,
         "voxel_mm": 1.0, "photons": 20_000, "gates": 1, "accum": 2, "normalized": False},
        # one member of a parameter study: an odd-sized heterogeneous volume, a Gaussian
        # beam, time gates, the normalised map
        {"name": "walk_ellipsoids_odd_1e6", "kind": "walk", "problem": "ellipsoids", "nx": 83, "ny": 61,
         "nz": 47, "voxel_mm": 0.8, "photons": 1_000_000, "gates": 3, "accum": 2, "normalized": True},
        # the headline workload (two spheres, ten gates, four detectors) at a tenth of its
        # photons, with the detected records that its user fits against
        {"name": "walk_spheres_detectors_1e7", "kind": "walk", "problem": "spheres", "nx": 64, "ny": 64,
         "nz": 64, "voxel_mm": 1.0, "photons": 10_000_000, "gates": 10, "accum": 2, "normalized": False},
        # layered tissue: the largest volume and map (3.4 GB), 50 gates, normalised
        {"name": "walk_layers_1e7", "kind": "walk", "problem": "layers", "nx": 256, "ny": 256, "nz": 128,
         "voxel_mm": 0.5, "photons": 10_000_000, "gates": 50, "accum": 2, "normalized": True},
        # the paper's B1 (photons end at the cube's surface) in the compensated FP32 mode
        {"name": "walk_b1_compensated_1e7", "kind": "walk", "problem": "b1", "nx": 60, "ny": 60, "nz": 60,
         "voxel_mm": 1.0, "photons": 10_000_000, "gates": 1, "accum": 1, "normalized": False},
        # the paper's B2a (Fresnel at the sphere and the surface)
        {"name": "walk_b2a_1e7", "kind": "walk", "problem": "b2a", "nx": 60, "ny": 60, "nz": 60,
         "voxel_mm": 1.0, "photons": 10_000_000, "gates": 1, "accum": 2, "normalized": False},
        # a host program that owns its device memory: the allocation-free call on unpadded
        # buffers of an odd size, no read-out
        {"name": "noalloc_ellipsoids_5e5", "kind": "noalloc", "problem": "ellipsoids", "nx": 57, "ny": 71,
         "nz": 53, "voxel_mm": 1.0, "photons": 500_000, "gates": 2, "accum": 2},
        # uneven simulations in one recorded launch, every map read back
        {"name": "batch_16", "kind": "batch", "sims": 16, "smallest": 32, "largest": 128, "photons": 400_000,
         "gates": 5},
        # denoising one map: the call at the end of a single low-photon run
        {"name": "denoise_apply_1", "kind": "apply", "volumes": 1, "nx": 64, "ny": 64, "nz": 64, "aux": 0},
        # denoising a set: the network alone on 16 encoded maps
        {"name": "denoise_forward_16", "kind": "forward", "volumes": 16, "nx": 64, "ny": 64, "nz": 64, "aux": 0},
        # a wide, ragged volume with the two medium features
        {"name": "denoise_forward_wide_aux", "kind": "forward", "volumes": 2, "nx": 128, "ny": 44, "nz": 36,
         "aux": 2},
        # one training step of the study's batch
        {"name": "denoise_train_4", "kind": "train", "volumes": 4, "nx": 64, "ny": 64, "nz": 64, "aux": 0},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["walk", "walk", "walk", "noalloc", "batch", "apply", "forward", "train"])
    if kind == "walk":
        problem = rng.choice(["cube", "spheres", "layers", "b1", "b2a", "ellipsoids", "ellipsoids"])
        case = {"kind": kind, "problem": problem, "accum": rng.choice([0, 1, 2, 2, 2]),
                "normalized": rng.random() < 0.5}
        case["voxel_mm"] = 0.5 if problem == "layers" else rng.choice([0.5, 0.8, 1.0])
        if problem == "ellipsoids":
            case |= {k: rng.randint(24, 110) for k in ("nx", "ny", "nz")}
            case["gates"] = rng.randint(1, 12)
        elif problem == "layers":
            case |= {"nx": rng.randint(64, 256), "ny": rng.randint(64, 256), "nz": rng.randint(48, 128)}
            case["gates"] = rng.randint(1, 50)
        else:
            side = {"cube": 64, "spheres": 64}.get(problem, 60)
            case |= {"nx": side, "ny": side, "nz": side, "voxel_mm": 1.0, "gates": GATES[problem][0]}
        # plain FP32 accumulation is for short runs: longer ones lose the hottest voxels' sums
        case["photons"] = int(min(_log(rng, 1e4, 1e6 if case["accum"] == 0 else 1e7), 1.4e12 / OPS[problem] / 2))
        return case
    if kind == "noalloc":
        return {"kind": kind, "problem": rng.choice(["cube", "ellipsoids"]), "nx": rng.randint(24, 110),
                "ny": rng.randint(24, 110), "nz": rng.randint(24, 110), "voxel_mm": rng.choice([0.5, 1.0]),
                "photons": int(_log(rng, 1e4, 3e6)), "gates": rng.randint(1, 8), "accum": rng.choice([0, 2])}
    if kind == "batch":
        return {"kind": kind, "sims": rng.randint(2, 24), "smallest": 32, "largest": rng.choice([64, 96, 128]),
                "photons": int(_log(rng, 2e4, 4e5)), "gates": rng.randint(1, 6)}
    nx = rng.choice([64, 64, 64, 128])
    case = {"kind": kind, "nx": nx, "ny": 4 * rng.randint(4, 24), "nz": 4 * rng.randint(4, 24),
            "aux": rng.choice([0, 0, 2])}
    room = int((2_000_000 if kind == "train" else 4_200_000) / (nx * case["ny"] * case["nz"]))
    case["volumes"] = max(1, min(room, int(_log(rng, 1, 17))))
    return case


# ------------------------------------------------------------------------- the problems
def _ellipsoids(rng, nz, ny, nx, n_inc=2):
    """Labels and media of a volume of random ellipsoids, drawn like the batched workloads."""
    media = [workloads.AIR]
    for _ in range(n_inc + 1):
        media.append((float(10 ** rng.uniform(-3, -1)), float(rng.uniform(0.5, 20.0)),
                      float(rng.uniform(0.5, 0.95)), float(rng.uniform(1.33, 1.45))))
    labels = np.ones((nz, ny, nx), dtype=np.uint8)
    z, y, x = np.ogrid[0:nz, 0:ny, 0:nx]
    for i in range(n_inc):
        c = rng.uniform(0.2, 0.8, size=3) * (nz, ny, nx)
        s = rng.uniform(0.1, 0.3, size=3) * (nz, ny, nx)
        labels[((z + 0.5 - c[0]) / s[0]) ** 2 + ((y + 0.5 - c[1]) / s[1]) ** 2 +
               ((x + 0.5 - c[2]) / s[2]) ** 2 <= 1.0] = i + 2
    return labels, np.array(media)


def _vary(media, rng):
    """The tissue rows' absorption and scattering within 5% of the workload's."""
    media = np.array(media, dtype=np.float64)
    media[1:, :2] *= rng.uniform(0.95, 1.05, size=media[1:, :2].shape)
    return media


def _problem(case, seed):
    """A workload of the case's kind and size, its optics and photon streams from the seed."""
    rng = np.random.default_rng(seed)
    nx, ny, nz, h = case["nx"], case["ny"], case["nz"], case["voxel_mm"]
    ph, gates, p = case["photons"], case["gates"], case["problem"]
    if p in ("cube", "spheres"):
        wl = workloads.c1() if p == "cube" else workloads.c2()
        if p == "cube" and (nz, ny, nx) != wl.labels.shape:
            wl = wl.with_(labels=np.ones((nz, ny, nx), dtype=np.uint8), src_pos=(nx * h / 2, ny * h / 2, 0.0))
        wl = wl.with_(media=_vary(wl.media, rng))
    elif p == "layers":
        labels = np.zeros((nz, ny, nx), dtype=np.uint8)
        workloads.paint_layers(labels, h, [3.0, 7.0, 2.0])
        media = [workloads.AIR, (0.019, 7.8, 0.89, 1.37), (0.019, 9.4, 0.89, 1.37),
                 (0.004, 0.01, 0.89, 1.37), (0.02, 6.6, 0.89, 1.37)]
        wl = workloads.Workload("layers", labels, h, _vary(media, rng), 1, (nx * h / 2, ny * h / 2, 0.0),
                                (0.0, 0.0, 1.0), 2.0, np.zeros((0, 4)), ph, gates, 0.1)
    elif p in ("b1", "b2a"):
        wl = workloads.paper_b(p.upper())
        wl = wl.with_(media=_vary(wl.media, rng))
    else:
        labels, media = _ellipsoids(rng, nz, ny, nx)
        pos = (float(rng.uniform(0.3, 0.7)) * nx * h, float(rng.uniform(0.3, 0.7)) * ny * h, 0.0)
        wl = workloads.Workload("ellipsoids", labels, h, media, 1, pos, (0.0, 0.0, 1.0), 1.5,
                                np.zeros((0, 4)), ph, gates, 1.0)
    dt = GATES[p][1] if p in GATES else 1.0
    return wl.with_(voxel_mm=h, n_photons=ph, n_gates=gates, dt_ns=dt, seed=1000 + int(seed))


# ------------------------------------------------------------------------- the network
LAYERS = [(16, 16), (16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (96, 32), (32, 32), (48, 16), (16, 16)]


def _params(rng, aux):
    """Weights of a working network: He-normal convolutions, small biases, a head that
    changes the map by a fraction of a unit, as a trained one does."""
    out = []
    for layer, (ci, co) in enumerate(LAYERS):
        fan = 27 * (1 + aux if layer == 0 else ci)
        w = rng.normal(size=(27, co, ci)) * math.sqrt(2.0 / fan)
        if layer == 0:
            w[:, :, 1 + aux:] = 0.0
        out += [w.ravel(), rng.normal(size=co) * 0.05]
    out += [rng.normal(size=16) * 0.05, rng.normal(size=1) * 0.05]
    return np.concatenate(out).astype(np.float32)


def _maps(case, seed):
    """Fluence maps (1/mm^2) of low-photon runs and their smooth counterparts: a beam's
    decay with the counting noise and the empty voxels of few photons."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    n, nz, ny, nx = case["volumes"], case["nz"], case["ny"], case["nx"]
    z = torch.arange(nz, device="cuda").view(1, nz, 1, 1) + 0.5
    y = torch.arange(ny, device="cuda").view(1, 1, ny, 1) + 0.5
    x = torch.arange(nx, device="cuda").view(1, 1, 1, nx) + 0.5
    r = torch.rand(n, 3, generator=gen, device="cuda")
    cx, cy = r[:, 0].view(n, 1, 1, 1) * nx, r[:, 1].view(n, 1, 1, 1) * ny
    mu = 0.08 + 0.3 * r[:, 2].view(n, 1, 1, 1)
    d = torch.sqrt((x - cx) ** 2 + (y - cy) ** 2 + (z - 1.0) ** 2) + 0.5
    clean = (0.1 * torch.exp(-mu * d) / d).contiguous()
    noisy = torch.poisson(clean * 1e6, generator=gen) * 1e-6
    aux = None
    if case["aux"]:
        lab = (torch.rand(n, case["aux"], 1, 1, 1, generator=gen, device="cuda") +
               0.3 * (torch.sin(0.1 * z + 0.15 * y + 0.05 * x) > 0).unsqueeze(1))
        aux = lab.expand(n, case["aux"], nz, ny, nx).contiguous()
    return noisy, clean, aux


def _network_inputs(case, seed):
    rng = np.random.default_rng(seed)
    p = _params(rng, case["aux"])
    noisy, clean, aux = _maps(case, seed)
    return p, noisy, clean, aux


# ------------------------------------------------------------------------- the contract
def prepare(case, seed):
    kind = case["kind"]
    if kind == "walk":
        wl = _problem(case, seed)
        sim = mcx.Simulation.from_workload(wl)
        out = torch.empty((wl.n_gates,) + wl.labels.shape, device="cuda")
        return {"case": case, "wl": wl, "sim": sim, "out": out}
    if kind == "noalloc":
        wl = _problem(case, seed)
        labels = torch.from_numpy(wl.labels).cuda()
        flu = torch.empty((wl.n_gates,) + wl.labels.shape, device="cuda",
                          dtype=torch.float64 if case["accum"] == 2 else torch.float32)
        tally = torch.empty(mcx.NOALLOC_NOUT, device="cuda", dtype=torch.float64)
        return {"case": case, "wl": wl, "labels": labels, "fluence": flu, "tally": tally}
    if kind == "batch":
        rng = np.random.default_rng(seed)
        batch, maps = mcx.Batch(), []
        for k in range(case["sims"]):
            sides = [s for s in (32, 48, 64, 96, 128) if case["smallest"] <= s <= case["largest"]]
            side = sides[k * 7 % len(sides)]
            labels, media = _ellipsoids(rng, side, side, side, 1 + k % 3)
            sx, sy = rng.uniform(0.0, side, size=2)
            n = int(round(case["photons"] * 10 ** rng.uniform(-1, 0)))
            batch.add(labels, 1.0, media, 0, (float(sx), float(sy), 0.0), (0.0, 0.0, 1.0), 0.0, n,
                      5000 + 100 * int(seed) + k)
            maps.append(torch.empty((case["gates"],) + labels.shape, device="cuda"))
        return {"case": case, "batch": batch, "maps": maps}
    p, noisy, clean, aux = _network_inputs(case, seed)
    shape = (case["nz"], case["ny"], case["nx"])
    net = mcx.Denoiser(shape, max_batch=case["volumes"], seed=0, n_aux=case["aux"])
    net.set_params(p)
    state = {"case": case, "net": net, "aux": aux, "out": torch.empty_like(noisy)}
    if kind == "apply":
        return state | {"phi": noisy}
    x, t = torch.empty_like(noisy), torch.empty_like(noisy)
    net.encode(noisy, x)
    net.encode(clean, t)
    net.sync()
    return state | {"x": x, "t": t}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "walk":
        wl, sim = state["wl"], state["sim"]
        det = len(wl.detectors) > 0
        sim.run(wl.n_photons, n_gates=wl.n_gates, dt_ns=wl.dt_ns, seed=wl.seed, reflect=wl.reflect,
                accum_mode=case["accum"], max_detected=1_000_000 if det else 0,
                stream=torch.cuda.current_stream())
        res = {"fluence": sim.fluence(normalized=case["normalized"], out=state["out"]), "tally": sim.tally()}
        if det:
            # as many records as a fit takes; about four times as many photons are detected
            rec, total = sim.detected(cap=wl.n_photons // 200)
            res |= {"detected": rec, "n_detected": total}
        return res
    if kind == "noalloc":
        wl = state["wl"]
        cfg = mcx.mcx_run_cfg_default(n_photons=wl.n_photons, n_gates=wl.n_gates, dt_ns=wl.dt_ns, seed=wl.seed,
                                      accum_mode=case["accum"], cuda_stream=torch.cuda.current_stream())
        mcx.mcx_run_noalloc(state["labels"], wl.voxel_mm, wl.media, wl.src_kind, wl.src_pos, wl.src_dir,
                            wl.waist_mm, cfg, state["fluence"], state["tally"])
        return {"fluence": state["fluence"], "tally": state["tally"]}
    if kind == "batch":
        b = state["batch"]
        b.run(n_gates=case["gates"], dt_ns=1.0, use_graph=1)
        for i, m in enumerate(state["maps"]):
            b.fluence(i, normalized=True, out=m)
        return {"maps": state["maps"], "tallies": [sum(b.tally(i).values()) for i in range(len(b))]}
    net = state["net"]
    if kind == "apply":
        net.apply(state["phi"], state["out"], aux=state["aux"])
        return state["out"]
    if kind == "forward":
        net.forward(state["x"], state["out"], aux=state["aux"])
        return state["out"]
    # the whole step, optimiser and weight refresh included, at a rate below the weights'
    # last bit, so that each pass starts from the same weights
    loss = net.train_step(state["x"], state["t"], 1e-30, aux=state["aux"])
    return {"loss": loss, "grads": net.grads()}


def work(case):
    kind = case["kind"]
    vox = case["nx"] * case["ny"] * case["nz"] if "nx" in case else 0
    if kind in ("walk", "noalloc"):
        map_bytes = vox * case["gates"] * (8 if kind == "noalloc" and case["accum"] == 2 else 4)
        return {"bytes": vox + map_bytes, "flops": case["photons"] * OPS[case["problem"]]}
    if kind == "batch":
        # photons are log-uniform over a factor of ten: their mean is 0.39 of the largest
        vox = case["sims"] * ((case["smallest"] + case["largest"]) / 2) ** 3
        return {"bytes": vox * (1 + 4 * case["gates"]),
                "flops": 0.39 * case["photons"] * case["sims"] * OPS["ellipsoids"]}
    n = case["volumes"] * vox
    per_voxel = 2.0 * 27 * ((1 + case["aux"]) * 16 + 16 * 16 + 48 * 16 + 16 * 16) + 32 + \
        2.0 * 27 * (16 * 32 + 32 * 32 + 96 * 32 + 32 * 32) / 8 + 2.0 * 27 * (32 * 64 + 64 * 64) / 64
    params = sum(27 * ci * co + co for ci, co in LAYERS) + 17
    if kind == "train":
        return {"bytes": n * 4 * (2 + case["aux"]) + params * 4 * 7, "flops": 3 * n * per_voxel}
    return {"bytes": n * 4 * (2 + case["aux"]) + params * 4, "flops": n * per_voxel}


# ------------------------------------------------------------------------- in 64 bits
def _conv(x, w, b, ci, co):
    k = w.view(3, 3, 3, co, ci).permute(3, 4, 0, 1, 2)
    return torch.relu(torch.nn.functional.conv3d(x, k, b, padding=1))


def _up(x):
    return x.repeat_interleave(2, 2).repeat_interleave(2, 3).repeat_interleave(2, 4)


def _network(p, x, aux):
    """The network on FP64 volumes [n, z, y, x]."""
    k, layers = 0, []
    for ci, co in LAYERS:
        layers.append((p[k:k + 27 * co * ci], p[k + 27 * co * ci:k + 27 * co * ci + co], ci, co))
        k += 27 * co * ci + co
    n, nz, ny, nx = x.shape
    a = torch.zeros((n, 16, nz, ny, nx), dtype=x.dtype, device=x.device)
    a = torch.cat([x.unsqueeze(1)] + ([aux] if aux is not None else []) +
                  [a[:, :15 - (0 if aux is None else aux.shape[1])]], 1)
    pool = torch.nn.functional.avg_pool3d
    s1 = _conv(_conv(a, *layers[0]), *layers[1])
    s2 = _conv(_conv(pool(s1, 2), *layers[2]), *layers[3])
    m = _conv(_conv(pool(s2, 2), *layers[4]), *layers[5])
    m = _conv(_conv(torch.cat([_up(m), s2], 1), *layers[6]), *layers[7])
    m = _conv(_conv(torch.cat([_up(m), s1], 1), *layers[8]), *layers[9])
    return x + torch.einsum("c,nczyx->nzyx", p[k:k + 16], m) + p[k + 16]


def exact(case, seed):
    if case["kind"] in ("walk", "noalloc", "batch"):
        return None                       # see the docstring
    p, noisy, clean, aux = _network_inputs(case, seed)
    p = torch.from_numpy(p).cuda().double()
    aux = None if aux is None else aux.double()

    def encode(phi):
        return (torch.log10(phi.double() + float(np.float32(1e-8))) + 4.0) / 2.0

    each = range(case["volumes"])         # one volume at a time, to bound the memory
    x = encode(noisy)
    if case["kind"] == "train":
        p.requires_grad_(True)
        t, total = encode(clean), 0.0
        for i in each:
            y = _network(p, x[i:i + 1], None if aux is None else aux[i:i + 1])
            loss = ((y - t[i:i + 1]) ** 2).sum() / x.numel()
            loss.backward()
            total += loss.detach()
        return {"loss": total, "grads": p.grad}
    with torch.no_grad():
        y = torch.cat([_network(p, x[i:i + 1], None if aux is None else aux[i:i + 1]) for i in each])
    if case["kind"] == "apply":
        return torch.clamp(10.0 ** (2.0 * y - 4.0) - float(np.float32(1e-8)), min=0.0)
    return y
