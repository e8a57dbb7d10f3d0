"""Workloads the framework's speed is measured on.

Every case is work a user has the framework do, through the public classes
``Simulator`` and ``Denoiser``:

  frame     one acquisition: ``trace`` of every transmit, then ``beamform`` to iq, envelope and dB
            (analytic, rough, meshed and convex scenes; plane, diverging, focused and
            synthetic-aperture transmits; transmit mixing)
  beamform  delay-and-sum of channel data that is already there (recorded, denoised, re-imaged)
  batch     several scenes x transmits in one ``batch_trace`` + ``batch_beamform`` (plan kept)
  adjoint   forward trace, then ``trace_adjoint`` (media and scatterer gradients)
  denoise   the U-Net's forward pass on channel data
  train     one training step of it (loss, gradient, Adam update)

Scenes, arrays and grids come from ``phantoms``; everything random comes from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2501_05828_gb300 as ur
import phantoms


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest call: one frame of the 32-element phantom (interactive use, unit tests)
        {"name": "frame_tiny", "kind": "frame", "scene": "tiny", "rays": 100_000, "scat": 200, "tx": "plane",
         "n_tx": 1, "span": 0.0, "nx": 128, "nz": 256},
        # a low-ray frame: the denoiser's input, a preview while a scene is edited; an odd image
        {"name": "frame_preview", "kind": "frame", "scene": "layered", "rays": 1_000_003, "scat": 30_000,
         "tx": "plane", "n_tx": 1, "span": 7.0, "nx": 383, "nz": 301},
        # the benchmarked RF frame: 1e7 rays, 50k scatterers, 0-degree plane wave
        {"name": "frame_layered", "kind": "frame", "scene": "layered", "rays": 10_000_000, "scat": 50_000,
         "tx": "plane", "n_tx": 1, "span": 0.0, "nx": 512, "nz": 256},
        # the paper's acquisition: rough bone in water, 25 plane waves, 12.8M rays
        {"name": "frame_paper", "kind": "frame", "scene": "paper", "rays": 512_000, "scat": 20_000, "tx": "plane",
         "n_tx": 25, "span": 30.0, "nx": 512, "nz": 256},
        # ultrafast imaging with diverging waves
        {"name": "frame_diverging", "kind": "frame", "scene": "layered", "rays": 500_000, "scat": 50_000,
         "tx": "diverging", "n_tx": 9, "span": 10.0, "nx": 512, "nz": 256},
        # the paper's bone as triangle meshes (5888 triangles), 25 plane waves
        {"name": "frame_mesh", "kind": "frame", "scene": "mesh", "rays": 256_000, "scat": 20_000, "tx": "plane",
         "n_tx": 25, "span": 30.0, "nx": 512, "nz": 256},
        # training-data generation: two scenes x 16 plane waves in one launch
        {"name": "batch_2x16", "kind": "batch", "scenes": 2, "scat": 60_000, "rays": 1_000_000, "n_tx": 16,
         "span": 15.0, "nx": 512, "nz": 256},
        # fitting tissue parameters: the forward trace and its adjoint
        {"name": "adjoint_layered", "kind": "adjoint", "rays": 4_000_000, "scat": 50_000, "n_tx": 1, "span": 0.0},
        # compounding 31 plane waves of the 128-element array
        {"name": "beamform_31", "kind": "beamform", "n_el": 128, "n_s": 3200, "fs": 40e6, "tx": "plane", "n_tx": 31,
         "span": 15.0, "nx": 512, "nz": 256, "radius": 0.0},
        # one convex-array frame on an odd grid
        {"name": "beamform_convex", "kind": "beamform", "n_el": 97, "n_s": 2999, "fs": 50e6, "tx": "diverging",
         "n_tx": 3, "span": 8.0, "nx": 311, "nz": 457, "radius": 0.05},
        # denoising the frames of one scene
        {"name": "denoise_4", "kind": "denoise", "batch": 4, "n_el": 128, "n_s": 3200},
        # training on traced pairs
        {"name": "train_8", "kind": "train", "batch": 8, "n_el": 128, "n_s": 3200},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "frame", "batch", "adjoint", "beamform", "beamform", "denoise",
                       "train"])
    img = {"nx": _log_int(rng, 96, 512), "nz": _log_int(rng, 96, 512)}
    if kind == "frame":
        scene = rng.choice(["tiny", "layered", "layered", "rough", "paper", "convex", "mesh"])
        n_tx = 1 if rng.random() < 0.4 else rng.randint(2, 25)
        tx = rng.choice(["plane", "plane", "plane", "diverging", "focused", "synthetic"])
        if scene == "convex" and tx == "plane":
            tx = "diverging"
        most = {"mesh": 6_400_000, "layered": 10_000_000}.get(scene, 8_000_000)
        total = _log_int(rng, 50_000, most)
        case = {"scene": scene, "rays": max(1000, total // n_tx), "scat": _log_int(rng, 200, 50_000), "tx": tx,
                "n_tx": n_tx, "span": round(rng.uniform(0.0, 30.0), 2)}
        if n_tx > 1 and rng.random() < 0.2:
            case["mix"] = True
        return {"kind": kind, **case, **img}
    if kind == "batch":
        n_tx = rng.randint(2, 16)
        return {"kind": kind, "scenes": rng.randint(1, 3), "scat": _log_int(rng, 10_000, 60_000),
                "rays": _log_int(rng, 50_000, 8_000_000 // n_tx), "n_tx": n_tx, "span": round(rng.uniform(1, 15), 2),
                **img}
    if kind == "adjoint":
        n_tx = rng.randint(1, 3)
        return {"kind": kind, "rays": _log_int(rng, 100_000, 4_000_000 // n_tx), "scat": _log_int(rng, 1000, 50_000),
                "n_tx": n_tx, "span": round(rng.uniform(0, 12), 2)}
    if kind == "beamform":
        radius = rng.choice([0.0, 0.0, 0.0, 0.05])
        return {"kind": kind, "n_el": _log_int(rng, 32, 192), "n_s": _log_int(rng, 800, 4096),
                "fs": rng.choice([25e6, 40e6, 50e6]), "tx": rng.choice(["plane", "plane", "diverging", "focused",
                                                                        "synthetic"]),
                "n_tx": _log_int(rng, 1, 25), "span": round(rng.uniform(0, 25), 2), **img, "radius": radius}
    n_el, n_s = 8 * rng.randint(4, 16), 8 * _log_int(rng, 40, 400)
    return {"kind": kind, "batch": rng.randint(1, 4), "n_el": n_el, "n_s": n_s}


# ------------------------------------------------------------------ inputs

def _transmits(kind, n_tx, span, n_el, pitch):
    """n_tx transmits of a kind, steered or placed over +-span degrees (Simulator.set_transmits' form)."""
    a = np.deg2rad(np.linspace(-span, span, n_tx) if n_tx > 1 else np.array([span]))
    aperture = n_el * pitch
    if kind == "diverging":
        return [(ur.TX_DIVERGING, float(np.float32(aperture * math.sin(t))),
                 float(np.float32(-0.5 * aperture * math.cos(t)))) for t in a]
    if kind == "focused":
        return [(ur.TX_FOCUSED, float(np.float32(0.03 * math.sin(t))), float(np.float32(0.03 * math.cos(t))))
                for t in a]
    if kind == "synthetic":
        return [(ur.TX_SYNTHETIC, float(int((k + 0.5) * n_el / n_tx)), 0.0) for k in range(n_tx)]
    return [(ur.TX_PLANE, float(np.float32(t)), 0.0) for t in a]


def _workload(case, seed):
    s, n = case["scene"], case["scat"]
    if s == "tiny":
        w = phantoms.tiny(seed=seed, n_scat=n)
    elif s in ("layered", "rough"):
        w = phantoms.layered(seed=seed, n_scat=n)
        if s == "rough":   # the bone's surface of the paper (GGX 0.5)
            w["scene"]["media"][3, 3] = 0.5
    elif s == "mesh":
        w = phantoms.paper_mesh_like(seed=seed, n_scat=n)
    else:
        w = phantoms.paper_like(seed=seed, n_scat=n, convex=s == "convex")
    A = w["array"]
    t = _transmits(case["tx"], case["n_tx"], case["span"], A["n_el"], A["pitch"])
    if case["tx"] == "plane":
        w["angles"] = np.array([q[1] for q in t], np.float32)
    else:
        w["transmits"] = t
    if case.get("mix"):
        w["mix"] = True
    z1 = 60e-3 if s in ("paper", "convex", "mesh") else None
    w["x_px"], w["z_px"] = phantoms.image_grid(A, case["nx"], case["nz"], z1=z1)
    return w


def _device(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _buffers(n, array):
    shape = (n, array["n_el"], array["n_s"])
    return torch.empty(shape, device="cuda"), torch.empty(shape, device="cuda")


def _echoes(gen, shape, f0, fs):
    """Speckle-like analytic channel data [..., n_s]: complex white noise through the 5-cycle pulse, decaying with
    depth, as rf and quad."""
    n_s = shape[-1]
    z = torch.randn(shape + (2,), generator=gen, device="cuda", dtype=torch.float32)
    f = torch.fft.fftfreq(n_s, 1.0 / fs, device="cuda", dtype=torch.float32)
    s = 5.0 / (4.0 * f0)
    band = torch.exp(-0.5 * (2 * math.pi * (f - f0) * s) ** 2)
    y = torch.fft.ifft(torch.fft.fft(torch.view_as_complex(z)) * band)
    y = y * torch.exp(-2.0 * torch.arange(n_s, device="cuda", dtype=torch.float32) / n_s)
    return y.real.contiguous(), y.imag.contiguous()


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _beamform_inputs(case, seed):
    """Array, transmits, pixel axes and channel data of a beamform case."""
    radius = case["radius"]
    pitch = np.deg2rad(70.0) * radius / case["n_el"] if radius else 0.3e-3
    A = phantoms.array_params(case["n_el"], case["n_s"], pitch=pitch, fs=case["fs"])
    if radius:
        A["radius"] = float(np.float32(radius))
    x, z = phantoms.image_grid(A, case["nx"], case["nz"])
    t = _transmits(case["tx"], case["n_tx"], case["span"], A["n_el"], A["pitch"])
    rf, quad = _echoes(_generator(seed), (case["n_tx"], A["n_el"], A["n_s"]), A["f0"], A["fs"])
    return A, t, x, z, rf, quad


# convolution layers of the U-Net in the order of the packed parameters: (name, c_in, c_out)
_CONV = [("e1a", 2, 32), ("e1b", 32, 32), ("e2a", 32, 64), ("e2b", 64, 64), ("e3a", 64, 128), ("e3b", 128, 128),
         ("e4a", 128, 256), ("e4b", 256, 256), ("d3a", 384, 128), ("d3b", 128, 128), ("d2a", 192, 64),
         ("d2b", 64, 64), ("d1a", 96, 32), ("d1b", 32, 32)]


def _network(seed):
    """He-normal weights [9, c_out, c_in] and small biases of every layer, and the 1x1 head, in float32."""
    rng = np.random.default_rng(seed)
    net = {n: ((rng.standard_normal((9, co, ci)) * math.sqrt(2.0 / (9 * ci))).astype(np.float32),
               (0.02 * rng.standard_normal(co)).astype(np.float32)) for n, ci, co in _CONV}
    net["head"] = ((0.15 * rng.standard_normal((2, 32))).astype(np.float32), np.zeros(2, np.float32))
    return net


def _pack(net):
    """The library's packed vector (ultraray.h): every tensor at a multiple of 8, the first layer's c_in padded to 32."""
    out = []
    for n, ci, co in _CONV:
        w, b = net[n]
        if n == "e1a":
            w = np.concatenate([w, np.zeros((9, co, 30), np.float32)], axis=2)
        out += [w.ravel(), b]
    out += [net["head"][0].ravel(), net["head"][1]]
    flat = np.concatenate(out)
    return np.concatenate([flat, np.zeros(-len(flat) % 8, flat.dtype)])


def _frames(case, seed):
    """Noisy channel data [batch, n_el, n_s] and, for training, its target."""
    g = _generator(seed)
    shape = (case["batch"], case["n_el"], case["n_s"])
    t = _echoes(g, shape, 5e6, 40e6)
    n = _echoes(g, shape, 5e6, 40e6)
    return [a + b for a, b in zip(t, n)] + list(t)


def prepare(case, seed):
    kind, seed = case["kind"], int(seed)
    if kind == "frame":
        w = _workload(case, seed)
        sim = ur.Simulator(0)
        sim.load(w)
        rf, quad = _buffers(case["n_tx"], w["array"])
        return {"kind": kind, "sim": sim, "w": w, "rf": rf, "quad": quad, "x": _device(w["x_px"]),
                "z": _device(w["z_px"]), "rays": case["rays"], "seed": seed}
    if kind == "batch":
        sim = ur.Simulator(0)
        for s in range(case["scenes"]):
            w = phantoms.layered(seed=seed + s, n_scat=case["scat"], z_fat=10e-3 + 0.5e-3 * s, bone_r=(4 + 2 * s) * 1e-3,
                                 angles_deg=np.linspace(-case["span"], case["span"], case["n_tx"]))
            sim.load(w, slot=s)
        x, z = phantoms.image_grid(w["array"], case["nx"], case["nz"])
        items = [(s, k, case["rays"], s * case["n_tx"] + k) for s in range(case["scenes"]) for k in range(case["n_tx"])]
        sim.batch_plan(items, x, z, capacity=case["rays"] * len(items) // 2 + 100_000)
        rf, quad = _buffers(len(items), w["array"])
        return {"kind": kind, "sim": sim, "w": w, "rf": rf, "quad": quad, "seed": seed}
    if kind == "adjoint":
        w = phantoms.layered(seed=seed, n_scat=case["scat"])
        n_tx = case["n_tx"]
        w["angles"] = np.array([q[1] for q in _transmits("plane", n_tx, case["span"], 128, 0.3e-3)], np.float32)
        sim = ur.Simulator(0)
        sim.load(w)
        rf, quad = _buffers(n_tx, w["array"])
        g_rf, g_quad = _echoes(_generator(seed), tuple(rf.shape), 5e6, 40e6)
        return {"kind": kind, "sim": sim, "w": w, "rf": rf, "quad": quad, "g": (g_rf, g_quad), "rays": case["rays"],
                "seed": seed}
    if kind == "beamform":
        A, t, x, z, rf, quad = _beamform_inputs(case, seed)
        sim = ur.Simulator(0)
        sim.set_array(A)
        sim.set_transmits(t)
        return {"kind": kind, "sim": sim, "rf": rf, "quad": quad, "x": _device(x), "z": _device(z)}
    net = ur.Denoiser(0, max_batch=case["batch"], n_el=case["n_el"], n_s=case["n_s"], seed=seed)
    net.set_params(_pack(_network(seed)))
    net.set_scale(0.5)
    return {"kind": kind, "net": net, "x": _frames(case, seed)}


def run(state):
    kind = state["kind"]
    if kind == "frame":
        sim, w, rf, quad = state["sim"], state["w"], state["rf"], state["quad"]
        sim.trace(state["rays"], state["seed"], w["max_bounces"], w["max_path"], rf=rf, quad=quad)
        iq, env, db = sim.beamform(rf, quad, state["x"], state["z"], w["dyn_range_db"])
        return {"rf": rf, "quad": quad, "iq": iq, "env": env, "db": db}
    if kind == "batch":
        sim, w, rf, quad = state["sim"], state["w"], state["rf"], state["quad"]
        sim.batch_trace(state["seed"], w["max_bounces"], w["max_path"], rf=rf, quad=quad)
        iq, env, db = sim.batch_beamform(rf, quad, w["dyn_range_db"], iq=True, env=True, db=True)
        return {"rf": rf, "quad": quad, "iq": iq, "env": env, "db": db}
    if kind == "adjoint":
        sim, w, rf, quad = state["sim"], state["w"], state["rf"], state["quad"]
        sim.trace(state["rays"], state["seed"], w["max_bounces"], w["max_path"], rf=rf, quad=quad)
        n_med, n_scat = len(w["scene"]["media"]), len(w["scene"]["scatterers"])
        gm, ga = sim.trace_adjoint(state["rays"], state["seed"], w["max_bounces"], *state["g"], max_path=w["max_path"],
                                   n_med=n_med, n_scat=n_scat)
        return {"rf": rf, "quad": quad, "grad_media": gm, "grad_amp": ga}
    if kind == "beamform":
        iq, env, db = state["sim"].beamform(state["rf"], state["quad"], state["x"], state["z"])
        return {"iq": iq, "env": env, "db": db}
    net, x = state["net"], state["x"]
    if kind == "denoise":
        return net.forward(x[0], x[1])
    # the learning rate at the end of the workflow's cosine decay (0.05 x 1e-3)
    loss, grad = net.train_step(x[0], x[1], x[2], x[3], 5e-5, grad=True)
    return {"loss": loss, "grad": grad}


# ------------------------------------------------------------------ what a pass cannot do without

# Per primary ray, from the tracer's counters on these scenes: straight segments, scatterer events at 50k
# (layered) or 20k (bone) scatterers, arrivals.  Operations per segment 40, interaction 72, event 38,
# connection 243, pulse tap 12 (the method's arithmetic, as the benchmark counts it).
_PER_RAY = {"tiny": (2.4, 0.0, 0.02), "layered": (3.7, 7.4, 0.23), "rough": (3.7, 7.4, 0.23),
            "paper": (2.5, 1.5, 0.03), "convex": (2.5, 1.5, 0.03), "mesh": (2.5, 1.5, 0.03)}


def _trace_flops(scene, rays, scat, n_s):
    seg, ev, arr = _PER_RAY[scene]
    ev *= scat / (50_000 if scene in ("layered", "rough") else 20_000)
    taps = 101 if n_s <= 3200 else 125
    return rays * (40 * seg + 72 * (seg - 1) + 38 * ev + 243 * 0.025 * ev + 12 * taps * arr)


def work(case):
    kind = case["kind"]
    if kind in ("frame", "batch", "adjoint"):
        scene = case.get("scene", "layered")
        n_el, n_s = (32, 1536) if scene == "tiny" else (128, 3200) if scene in ("layered", "rough") else (128, 4096)
        n_tx = case["n_tx"] * case.get("scenes", 1)
        chan = 2 * 4 * n_tx * n_el * n_s
        scat = 16 * case["scat"] * case.get("scenes", 1)
        flops = _trace_flops(scene, case["rays"] * n_tx, case["scat"], n_s)
        if kind == "adjoint":   # each arrival's path and pulse again, with their derivatives
            return {"bytes": 2 * chan + 2 * scat, "flops": 3 * flops}
        px = case["nx"] * case["nz"]
        das = 14 * px * n_el * n_tx   # receive delay shared by the transmits: add, split, 4 lerp multiply-adds, sum
        return {"bytes": 2 * chan + scat + 16 * px * case.get("scenes", 1), "flops": flops + das}
    if kind == "beamform":
        px, n = case["nx"] * case["nz"], case["n_tx"] * case["n_el"]
        return {"bytes": 8 * n * case["n_s"] + 16 * px, "flops": 14 * px * n}
    p = case["batch"] * case["n_el"] * case["n_s"]
    scale = {"e1": 1, "e2": 4, "e3": 16, "e4": 64, "d3": 16, "d2": 4, "d1": 1}
    fwd = sum(18 * ci * co * p / scale[n[:2]] for n, ci, co in _CONV)
    weights = 4 * sum(9 * ci * co for _, ci, co in _CONV)
    if kind == "denoise":
        return {"bytes": 16 * p + weights / 2, "flops": fwd}
    return {"bytes": 16 * p + 6 * weights, "flops": 3 * fwd}


# ------------------------------------------------------------------ the same in 64 bits

def _das64(A, t, x, z, rf, quad, dyn_range_db=60.0):
    dev = rf.device
    f8 = lambda v: torch.as_tensor(np.asarray(v, np.float64), device=dev)
    n_el, n_s, q, R = A["n_el"], A["n_s"], A["fs"] / A["c_bf"], A.get("radius", 0.0)
    k = np.arange(n_el) - 0.5 * (n_el - 1)
    cx = R * np.sin(k * A["pitch"] / R) if R else k * A["pitch"]
    cz = R * (np.cos(k * A["pitch"] / R) - 1.0) if R else 0.0 * k
    X, Z = f8(x)[None, :], f8(z)[:, None]
    sr = torch.zeros((len(z), len(x)), dtype=torch.float64, device=dev)
    si = torch.zeros_like(sr)
    rx = [torch.sqrt((X - cx[e]) ** 2 + (Z - cz[e]) ** 2) for e in range(n_el)]
    for j, (kind, a, b) in enumerate(t):
        if kind == ur.TX_PLANE:
            T = X * math.sin(a) + Z * math.cos(a) - float(np.min(cx * math.sin(a) + cz * math.cos(a)))
        else:
            vx, vz = (cx[int(a)], cz[int(a)]) if kind == ur.TX_SYNTHETIC else (a, b)
            r, re = torch.sqrt((X - vx) ** 2 + (Z - vz) ** 2), np.hypot(cx - vx, cz - vz)
            if kind == ur.TX_FOCUSED:
                T = float(re.max()) + torch.where(Z >= vz, r, -r)
            else:
                T = r - float(re.min())
        for e in range(n_el):
            tau = (T + rx[e]) * q
            ok = (tau >= 0) & (tau <= n_s - 1)
            i0 = tau.floor().clamp(0, n_s - 1)
            f, i0 = tau - i0, i0.long()
            i1 = (i0 + 1).clamp(max=n_s - 1)
            for src, acc in ((rf, sr), (quad, si)):
                row = src[j, e].double()
                acc += torch.where(ok, row[i0] * (1 - f) + row[i1] * f, 0.0)
    env = torch.sqrt(sr * sr + si * si)
    db = torch.clamp(20.0 * torch.log10(env / env.max()), min=-dyn_range_db)
    return {"iq": torch.stack([sr, si], -1), "env": env, "db": db}


def _unet64(p, x):
    F = torch.nn.functional

    def block(n, v):
        for s in "ab":
            v = F.relu(F.conv2d(v, p[n + s + ".w"], p[n + s + ".b"], padding=1))
        return v

    up = lambda v: v.repeat_interleave(2, 2).repeat_interleave(2, 3)
    e1 = block("e1", x)
    e2 = block("e2", F.avg_pool2d(e1, 2))
    e3 = block("e3", F.avg_pool2d(e2, 2))
    e4 = block("e4", F.avg_pool2d(e3, 2))
    d3 = block("d3", torch.cat([up(e4), e3], 1))
    d2 = block("d2", torch.cat([up(d3), e2], 1))
    d1 = block("d1", torch.cat([up(d2), e1], 1))
    return x + F.conv2d(d1, p["head.w"], p["head.b"])


def exact(case, seed):
    kind = case["kind"]
    if kind == "beamform":
        return _das64(*_beamform_inputs(case, int(seed)))
    if kind not in ("denoise", "train"):
        return None   # a Monte Carlo trace has no value in plain torch: its paths are the tracer's own
    net = _network(int(seed))
    p = {}
    for n, ci, co in _CONV:
        w = net[n][0].reshape(3, 3, co, ci).transpose(2, 3, 0, 1)
        p[n + ".w"] = _device(w.astype(np.float64))
        p[n + ".b"] = _device(net[n][1].astype(np.float64))
    p["head.w"] = _device(net["head"][0].astype(np.float64).reshape(2, 32, 1, 1))
    p["head.b"] = _device(net["head"][1].astype(np.float64))
    scale = 0.5
    fr = [v.double() / scale for v in _frames(case, int(seed))]
    if kind == "denoise":
        with torch.no_grad():
            y = torch.cat([_unet64(p, torch.stack([fr[0][k:k + 1], fr[1][k:k + 1]], 1))
                           for k in range(case["batch"])])
        return [y[:, 0] * scale, y[:, 1] * scale]
    for v in p.values():
        v.requires_grad_(True)
    loss, n = 0.0, 2 * fr[0].numel()
    for k in range(case["batch"]):
        y = _unet64(p, torch.stack([fr[0][k:k + 1], fr[1][k:k + 1]], 1))
        d = y - torch.stack([fr[2][k:k + 1], fr[3][k:k + 1]], 1)
        part = (d * d).sum() / n
        part.backward()
        loss += float(part)
    g = {}
    for n, ci, co in _CONV:
        g[n] = (p[n + ".w"].grad.permute(2, 3, 0, 1).reshape(9, co, ci).cpu().numpy(), p[n + ".b"].grad.cpu().numpy())
    g["head"] = (p["head.w"].grad.reshape(2, 32).cpu().numpy(), p["head.b"].grad.cpu().numpy())
    return {"loss": loss, "grad": _device(_pack(g))}
