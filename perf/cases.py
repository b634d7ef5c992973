"""Performance cases: the work a user of the library has it do, through the Python binding.

``listed()`` names the cases that are always measured, ``draw(rng)`` gives further ones
over the same ranges, ``prepare(case, seed)`` makes what a user's program holds before
the call (models resident on the GPU, run description, output buffers), ``run(state)``
is one pass (step 1, then the images of every camera), ``work(case)`` what a pass
cannot do without, ``exact(case, seed)`` the outputs in 64 bits where they have a
closed form.

Sizes are those of the repository's tests and of bench.py: the Rayleigh sphere, the
dichroic slab, the flared disk (plain and refined), the plane-parallel slab, the
aligned-spheroid sphere, the batched sweep and the network surrogate.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2512_01283_gb300 import mcrt as M
from paper_2512_01283_gb300 import workloads as W

DEV = "cuda"


# ----------------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: a quick look at a small Rayleigh sphere, where launches count
        {"name": "sphere32", "kind": "sphere", "n": 32, "tau": 1.0, "packets": 100_000, "cams": 1, "npix": 64},
        # pure absorption: a beam through aligned grains, and the slab's own emission
        {"name": "slab64", "kind": "slab", "n": 64, "tau": 1.0, "packets": 1_000_000, "cams": 1, "npix": 64,
         "up": True},
        # the FP64 instantiation, as used to check an FP32 result
        {"name": "disk24_fp64", "kind": "disk", "n": 24, "tau": 1000.0, "packets": 100_000, "cams": 4, "npix": 32,
         "precision": "fp64"},
        # a test-sized disk: star and thermal packets, eight cameras
        {"name": "disk64", "kind": "disk", "n": 64, "tau": 1000.0, "packets": 1_000_000, "cams": 8, "npix": 64,
         "precision": "fp32"},
        # the same from host arrays to host images: upload, both steps, download
        {"name": "disk64_host", "kind": "disk_host", "n": 64, "tau": 1000.0, "packets": 1_000_000, "cams": 8,
         "npix": 64},
        # the benchmark's disk: the largest production run
        {"name": "disk192", "kind": "disk", "n": 192, "tau": 1000.0, "packets": 100_000_000, "cams": 8, "npix": 256,
         "precision": "fp32"},
        # the benchmark's composite grid: root grid and a refined inner patch
        {"name": "refined128", "kind": "refined", "n": 128, "factor": 4, "packets": 10_000_000, "cams": 8,
         "npix": 256},
        # the benchmark's atmosphere: periodic axes, many scatterings per packet
        {"name": "plane_parallel", "kind": "plane", "n": 64, "nz": 128, "tau": 10.0, "packets": 10_000_000,
         "cams": 2, "npix": 64},
        # the benchmark's aligned spheroids
        {"name": "spheroids128", "kind": "spheroids", "n": 128, "tau": 1.0, "packets": 10_000_000, "cams": 2,
         "npix": 256},
        # a parameter sweep: clumpy models at several wavelengths in one batched launch
        {"name": "sweep32", "kind": "sweep", "models": 4, "wavelengths": 8, "n_min": 32, "n_max": 192,
         "packets": 500_000, "npix": 128},
        # grain optics from the trained network
        {"name": "surrogate64", "kind": "surrogate", "n": 64, "tau": 1000.0, "packets": 500_000, "cams": 8,
         "npix": 64},
        # one forward and backward pass of the network on a user's own samples
        {"name": "network_grad", "kind": "grad", "batch": 2048},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["sphere", "slab", "disk", "disk", "disk_host", "refined", "plane", "spheroids", "sweep",
                       "surrogate", "grad"])
    cams = rng.randint(1, 8)
    if kind == "sphere":
        return {"kind": kind, "n": int(_log(rng, 16, 128)), "tau": _log(rng, 0.1, 10.0),
                "packets": int(_log(rng, 2e4, 1e7)), "cams": cams, "npix": int(_log(rng, 32, 256))}
    if kind == "slab":
        return {"kind": kind, "n": int(_log(rng, 16, 128)), "tau": _log(rng, 0.1, 30.0),
                "packets": int(_log(rng, 1e5, 1e7)), "cams": 1, "npix": int(_log(rng, 32, 256)),
                "up": rng.random() < 0.5}
    if kind in ("disk", "disk_host"):
        fp64 = kind == "disk" and rng.random() < 0.2
        hi = 2e5 if fp64 else (5e7 if kind == "disk" else 1e7)
        case = {"kind": kind, "n": int(_log(rng, 24, 192)), "tau": _log(rng, 1.0, 1000.0),
                "packets": int(_log(rng, 5e4, hi)), "cams": cams, "npix": int(_log(rng, 32, 256))}
        if kind == "disk":
            case["precision"] = "fp64" if fp64 else "fp32"
        return case
    if kind == "refined":
        return {"kind": kind, "n": 16 * rng.randint(2, 8), "factor": rng.randint(2, 4),
                "packets": int(_log(rng, 1e5, 1e7)), "cams": cams, "npix": int(_log(rng, 32, 256))}
    if kind == "plane":
        return {"kind": kind, "n": int(_log(rng, 4, 96)), "nz": int(_log(rng, 16, 160)), "tau": _log(rng, 1.0, 10.0),
                "packets": int(_log(rng, 1e5, 1e7)), "cams": cams, "npix": int(_log(rng, 32, 128))}
    if kind == "spheroids":
        return {"kind": kind, "n": int(_log(rng, 16, 128)), "tau": _log(rng, 0.01, 10.0),
                "packets": int(_log(rng, 1e5, 1e7)), "cams": cams, "npix": int(_log(rng, 32, 256))}
    if kind == "sweep":
        return {"kind": kind, "models": rng.randint(1, 6), "wavelengths": rng.randint(2, 8), "n_min": 32,
                "n_max": rng.randint(48, 192), "packets": int(_log(rng, 2e4, 5e5)), "npix": rng.randint(24, 128)}
    if kind == "surrogate":
        return {"kind": kind, "n": int(_log(rng, 24, 128)), "tau": _log(rng, 10.0, 1000.0),
                "packets": int(_log(rng, 2e4, 5e5)), "cams": cams, "npix": int(_log(rng, 32, 128))}
    return {"kind": kind, "batch": int(_log(rng, 512, 8192))}


# ----------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------
@functools.lru_cache(maxsize=3)
def _disk_base(n, tau):
    return W.disk(n=n, tau_mid=tau)


@functools.lru_cache(maxsize=2)
def _refined_base(n, factor):
    return W.disk_refined(n=n, factor=factor)


def _rng(seed):
    return np.random.default_rng([seed & 0xffffffff, 1283])


def _to_gpu(model, scale):
    """The model with its fields as CUDA tensors, the opacities times ``scale``."""
    out = dict(model)
    for key in ("kappa_abs", "kappa_sca", "bfield", "emissivity"):
        if model.get(key) is not None:
            out[key] = torch.from_numpy(np.ascontiguousarray(model[key])).to(DEV)
            if key.startswith("kappa"):
                out[key] = out[key] * scale
    if model.get("refine"):
        out["refine"] = [_to_gpu(q, scale) for q in model["refine"]]
    return out


def _scale(seed):
    """Opacity factor of a seed's model: seeds differ in the medium and in the packets."""
    return float(np.float32(_rng(seed).uniform(0.9, 1.1)))


def _side_cameras(n_cam, npix, fov, center=None):
    """Cameras around the object, off the grid axes but for the first two."""
    dirs = [(1.0, 0.0, 0.0), (0.0, 0.0, 1.0)]
    for k in range(n_cam - 2):
        a, i = 0.37 + 0.9 * k, 0.4 + 0.3 * k
        dirs.append((math.sin(i) * math.cos(a), math.sin(i) * math.sin(a), math.cos(i)))
    return [W.camera(d, (npix, npix), (fov, fov), center) for d in dirs[:n_cam]]


def _seeded(run, seed):
    return dict(run, seed=int(_rng(seed).integers(1, 1 << 31)))


def _scene(case, seed):
    """Model (host arrays) and run of a case."""
    kind, cams, npix = case["kind"], case.get("cams", 1), case.get("npix", 64)
    n, packets = case.get("n"), case.get("packets")
    if kind == "sphere":
        model = W.rayleigh_sphere(n=n, tau=case["tau"])
        run = dict(W.rayleigh_sphere_run(packets, npix=npix), cameras=_side_cameras(cams, npix, 2.0))
    elif kind == "slab":
        model = W.dichroic_slab(n=n, tau=case["tau"], emissivity=1.0)
        run = W.beam_run(packets, direction=1 if case["up"] else -1,
                         cameras=[W.camera((0.0, 0.0, 1.0), (npix, npix), (1.0, 1.0))])
    elif kind in ("disk", "disk_host", "surrogate"):
        model, run = _disk_base(n, case["tau"]), W.disk_run(packets, n_cam=cams, npix=npix)
    elif kind == "refined":
        model, run = _refined_base(n, case["factor"]), W.disk_run(packets, n_cam=cams, npix=npix)
    elif kind == "plane":
        model = W.plane_parallel_slab(nxy=n, nz=case["nz"], tau=case["tau"], albedo=0.9, periodic=3,
                                      b_angle_deg=30.0, p=0.05)
        run = W.center_source_run(packets, cameras=_side_cameras(cams, npix, 1.0))
    else:  # spheroids
        model = W.spheroid_sphere(n=n, tau=case["tau"], albedo=0.5)
        run = {"sources": [{"type": "point", "pos": (0.0, 0.0, 0.0), "luminosity": 1.0, "n_packets": packets}],
               "cameras": _side_cameras(cams, npix, 2.0), "roulette_threshold": 1e-4, "roulette_survival": 0.1}
    return model, _seeded(run, seed)


def _clumpy(n, seed):
    """Log-normal density of the sweep (white noise smoothed over 2 cells), on the GPU."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    g = torch.randn(n, n, n, generator=gen, device=DEV)
    f = torch.fft.fftfreq(n, device=DEV)
    w = torch.exp(-2.0 * (math.pi * 2.0 * f) ** 2)
    g = torch.fft.ifftn(torch.fft.fftn(g) * w[:, None, None] * w[None, :, None] * w[None, None, :]).real
    g = (g - g.mean()) / g.std()
    return torch.exp(g - 0.5)


def _sweep_models(case, seed):
    rng = _rng(seed)
    lams = np.logspace(np.log10(0.5), np.log10(3.0), case["wavelengths"])
    optics = W.table_optics()
    out = []
    for m in range(case["models"]):
        # edges spread over the range, the same for every seed
        n = case["n_min"] + (case["n_max"] - case["n_min"]) * (m + 1) // case["models"]
        tau = 10 ** (2.0 * (m + rng.uniform(0.4, 0.6)) / case["models"])
        rho = _clumpy(n, int(rng.integers(1 << 30)))
        for lam in lams:
            kext = (float(tau / 2.0 * lam ** -1.5) * rho).contiguous()
            ks = 0.6 * kext
            out.append({"lo": (-1.0, -1.0, -1.0), "hi": (1.0, 1.0, 1.0), "kappa_abs": kext - ks, "kappa_sca": ks,
                        "bfield": None, "emissivity": None, "optics": optics})
    return out


def _net_inputs(gen, n):
    d = torch.randn(2, n, 3, generator=gen, device=DEV)
    d = d / d.norm(dim=2, keepdim=True)
    s = 2.0 * torch.rand(n, 1, generator=gen, device=DEV) - 1.0
    return torch.cat([d[0], d[1], s], dim=1)


def _net_forward(layers, u):
    x = torch.zeros(u.shape[0], layers[0][0].shape[1], device=u.device, dtype=u.dtype)
    x[:, :u.shape[1]] = u
    for i, (w, b) in enumerate(layers):
        x = torch.nn.functional.linear(x, w, b)
        if i + 1 < len(layers):
            x = torch.nn.functional.silu(x)
    return x[:, :M.Surrogate.N_OUT]


@functools.lru_cache(maxsize=1)
def _trained_layers():
    """Weights of the surrogate of the disk's tables, as a user who trained it once has
    them on disk: fitted here with plain PyTorch (seeded), so that every process that
    measures a case runs the same network.  The network does not depend on the disk."""
    model = M.Model(W.disk(n=16))
    sur = M.Surrogate(model, seed=11)
    gen = torch.Generator(device=DEV).manual_seed(1283)
    layers = [[torch.from_numpy(np.array(w)).to(DEV), torch.from_numpy(np.array(b)).to(DEV)]
              for w, b in sur.get_params()]
    params = [t.requires_grad_() for layer in layers for t in layer]
    opt = torch.optim.Adam(params, lr=3e-3, fused=True)
    steps, batch = 2500, 8192
    sched = torch.optim.lr_scheduler.CosineAnnealingLR(opt, steps, eta_min=1.5e-4)
    pool = _net_inputs(gen, 1 << 20)
    labels = torch.from_numpy(sur.labels(pool.cpu().numpy())).to(DEV)
    for it in range(steps):
        at = (it * batch) % (1 << 20)
        opt.zero_grad(set_to_none=True)
        loss = torch.mean((_net_forward(layers, pool[at:at + batch]) - labels[at:at + batch]) ** 2)
        loss.backward()
        opt.step()
        sched.step()
    out = [(w.detach().cpu().numpy(), b.detach().cpu().numpy()) for w, b in layers]
    sur.close()
    model.close()
    return out


class _State:
    """What a user's program holds: the model(s), the run description, output buffers."""

    def __init__(self, **kw):
        self.__dict__.update(kw)

    def __del__(self):
        for name in ("batch", "sur", "model"):
            if getattr(self, name, None) is not None:
                getattr(self, name).close()
        for m in getattr(self, "models", None) or []:
            m.close()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "grad":
        model = M.Model(W.disk(n=16))
        sur = M.Surrogate(model, seed=3 + seed % 1000)
        rng = _rng(seed)
        d = rng.standard_normal((2, case["batch"], 3))
        d /= np.linalg.norm(d, axis=2, keepdims=True)
        u = np.concatenate([d[0], d[1], rng.uniform(-1, 1, (case["batch"], 1))], axis=1).astype(np.float32)
        return _State(kind=kind, model=model, sur=sur, u=u, t=sur.labels(u))
    if kind == "sweep":
        models = [M.Model(m) for m in _sweep_models(case, seed)]
        run = W.sweep_run(n_packets=case["packets"], npix=case["npix"])
        batch = M.Batch(models, run)
        npix = case["npix"]
        images = torch.zeros(len(models), len(run["cameras"]), 4, npix, npix, dtype=torch.float64, device=DEV)
        return _State(kind=kind, models=models, batch=batch, seed=_seeded(run, seed)["seed"], images=images)
    host, run = _scene(case, seed)
    npix, cams = case["npix"], len(run["cameras"])
    if kind == "disk_host":
        s = np.float32(_scale(seed))
        host = dict(host, kappa_abs=host["kappa_abs"] * s, kappa_sca=host["kappa_sca"] * s)
        # pinned host memory, as bench.py's end-to-end line holds its model
        for key in ("kappa_abs", "kappa_sca", "bfield", "emissivity"):
            host[key] = torch.from_numpy(np.ascontiguousarray(host[key])).pin_memory().numpy()
        images = torch.zeros(cams, 4, npix, npix, dtype=torch.float64).pin_memory().numpy()
        return _State(kind=kind, host=host, run=run, images=images, absorbed=np.zeros(host["kappa_abs"].shape))
    model = M.Model(_to_gpu(host, 1.0 if kind == "slab" else _scale(seed)))
    images = torch.zeros(cams, 4, npix, npix, dtype=torch.float64, device=DEV)
    absorbed = torch.zeros(model.ncell, dtype=torch.float64, device=DEV)
    sur = None
    optics = "tables"
    if kind == "surrogate":
        sur = M.Surrogate(model, seed=11)
        sur.set_params(_trained_layers())
        model.set_surrogate(sur)
        optics = "surrogate"
    return _State(kind=kind, model=model, sur=sur, run=run, images=images, absorbed=absorbed, optics=optics,
                  precision=case.get("precision", "fp32"))


# ----------------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------------
COUNTS = ("events", "segments", "scatterings", "emitted", "escaped", "roulette_killed", "trials")
ENERGIES = ("emitted_energy", "escaped_energy", "absorbed_energy", "roulette_lost", "roulette_gain")


def _totals(st):
    return {"counts": np.array([int(st[k]) for k in COUNTS]), "energies": np.array([st[k] for k in ENERGIES])}


def run(state):
    if state.kind == "grad":
        loss, layers = state.sur.grad(state.u, state.t)
        return {"loss": loss, "grads": [a for layer in layers for a in layer]}
    if state.kind == "sweep":
        st = state.batch.launch(state.seed)
        return dict(_totals(st), images=state.batch.images(state.images))
    if state.kind == "disk_host":
        model = M.Model(state.host)
        st = M.launch(model, state.run)
        for k in range(len(state.images)):
            model.image(k, state.images[k])
        model.tallies_into(absorbed=state.absorbed)
        model.close()
    else:
        st = M.launch(state.model, state.run, precision=state.precision, optics=state.optics)
        for k in range(len(state.images)):
            state.model.image(k, state.images[k])
        state.model.tallies_into(absorbed=state.absorbed)
    return dict(_totals(st), images=state.images, absorbed=state.absorbed)


# ----------------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------------
# Segments, tallying segments and scatterings of a packet: per cell of the grid's edge
# (a path crosses a number of cells proportional to it) and per packet, measured at the
# listed sizes; and operations of the method's formulas (a segment's distance, frame
# rotation and in-cell transfer; a camera's matrix, plane rotation and product; one
# scattering with its trials).
PER_EDGE = {"sphere": (1.28, 1.09, 1.5), "slab": (1.0, 0.0, 0.0), "disk": (0.57, 0.37, 8.4),
            "refined": (0.88, 0.52, 8.4), "plane": (4.6, 4.6, 41.0), "spheroids": (1.09, 0.90, 0.63),
            "sweep": (1.12, 1.12, 6.2)}
FLOP_SEGMENT, FLOP_CAMERA, FLOP_SCATTER = 150.0, 80.0, 400.0
FLOP_NET = 2.0 * (7 * 128 + 3 * 128 * 128 + 128 * 20)


def _grid_cells(case):
    kind = case["kind"]
    if kind == "plane":
        return case["n"] ** 2 * case["nz"], max(case["n"], case["nz"])
    if kind == "refined":
        n, f = case["n"], case["factor"]
        return n ** 3 + (n // 4) ** 2 * (n // 8) * f ** 3, n
    return case["n"] ** 3, case["n"]


def work(case):
    kind = case["kind"]
    if kind == "grad":
        b = case["batch"]
        params = 16 * 128 + 3 * 128 * 128 + 128 * 24 + 4 * 128 + 24
        return {"bytes": 4.0 * (b * 27 + 2 * params), "flops": 3.0 * FLOP_NET * b}
    if kind == "sweep":
        total = {"bytes": 0.0, "flops": 0.0}
        for m in range(case["models"]):
            n = case["n_min"] + (case["n_max"] - case["n_min"]) * (m + 1) // case["models"]
            one = _mc_work("sweep", n ** 3, n, case["packets"], 1, case["npix"], 8, False)
            for k in total:
                total[k] += case["wavelengths"] * one[k]
        return total
    cells, edge = _grid_cells(case)
    key = "disk" if kind in ("disk_host", "surrogate") else kind
    fields = {"sphere": 8, "slab": 24, "plane": 20, "spheroids": 20}.get(kind, 24)
    return _mc_work(key, cells, edge, case["packets"], case["cams"], case["npix"], fields, kind == "surrogate")


def _mc_work(key, cells, edge, packets, cams, npix, field_bytes, network):
    """Every field read once, the source and absorbed tallies and the images written once."""
    seg, tal, sca = PER_EDGE[key]
    rows = packets * edge * tal * cams
    flops = packets * (edge * seg * FLOP_SEGMENT + sca * FLOP_SCATTER) + rows * FLOP_CAMERA
    flops += cams * npix * npix * edge * FLOP_SEGMENT
    if network:
        flops += (rows + packets * sca) * FLOP_NET
    return {"bytes": float(cells * (field_bytes + 32 * cams + 8) + cams * npix * npix * 32), "flops": float(flops)}


# ----------------------------------------------------------------------------------
# the same in 64 bits
# ----------------------------------------------------------------------------------
def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 (Salmon et al. 2011) on arrays of counters."""
    mask = np.uint64(0xffffffff)
    c = [np.asarray(v, dtype=np.uint64) & mask for v in (c0, c1, c2, c3)]
    k0, k1 = int(k0), int(k1)
    for r in range(10):
        a = np.uint64(0xD2511F53) * c[0]
        b = np.uint64(0xCD9E8D57) * c[2]
        kr0 = np.uint64((k0 + r * 0x9E3779B9) & 0xffffffff)
        kr1 = np.uint64((k1 + r * 0xBB67AE85) & 0xffffffff)
        c = [(b >> np.uint64(32)) ^ c[1] ^ kr0, b & mask, (a >> np.uint64(32)) ^ c[3] ^ kr1, a & mask]
    return c


def _exact_slab(case, seed):
    """A beam through an absorbing slab of aligned grains: I and Q decay as
    e^{-t} (cosh, -sinh)(alpha2 t); a packet's column comes from its random numbers; seen
    from above the slab shows its own emission, (1 - e^{-K tau}) (B, 0)."""
    n, tau, packets, npix = case["n"], float(np.float32(case["tau"])), case["packets"], case["npix"]
    run_ = _scene(dict(case, n=2), seed)[1]
    a2 = float(np.float32(-0.05))
    pid = np.arange(packets, dtype=np.uint64)
    zero = np.zeros_like(pid)
    x = _philox(pid, zero, zero, zero + np.uint64(1), run_["seed"], 0)
    u = [((v >> np.uint64(8)) | np.uint64(1)).astype(np.float64) * 2.0 ** -24 for v in x[:2]]
    col = np.bincount(np.floor(u[1] * n).astype(np.int64) * n + np.floor(u[0] * n).astype(np.int64), minlength=n * n)
    t = tau * np.arange(n + 1) / n
    level = np.exp(-t) * np.cosh(a2 * t)
    drop = level[:-1] - level[1:]
    if not case["up"]:
        drop = drop[::-1]
    absorbed = (drop[:, None] * (col / packets)[None, :]).reshape(-1)
    images = np.zeros((1, 4, npix, npix))
    images[0, 0] = 1.0 - level[-1]
    images[0, 1] = np.exp(-tau) * np.sinh(a2 * tau)
    energies = np.array([1.0, level[-1], 1.0 - level[-1], 0.0, 0.0])
    return {"counts": None, "energies": energies, "images": images, "absorbed": absorbed}


def _exact_grad(case, seed):
    """Loss and gradients of the network by automatic differentiation in FP64."""
    state = prepare(case, seed)
    layers = [[torch.from_numpy(np.array(w)).to(DEV, torch.float64).requires_grad_() for w in layer]
              for layer in state.sur.get_params()]
    u, t = (torch.from_numpy(v).to(DEV, torch.float64) for v in (state.u, state.t))
    loss = torch.mean((_net_forward(layers, u) - t) ** 2)
    loss.backward()
    return {"loss": float(loss.detach()), "grads": [w.grad for layer in layers for w in layer]}


def exact(case, seed):
    if case["kind"] == "slab":
        return _exact_slab(case, seed)
    if case["kind"] == "grad":
        return _exact_grad(case, seed)
    # a Monte-Carlo run has no closed form, and a 64-bit one in numpy takes far longer than seconds
    return None
