"""The workloads whose speed counts, each through the calls a user's program makes.

Kinds of case:
  lb       one simulation: steps, then the fields (phi, rho, u) on the device, as a run with
           snapshots does.  Storages, collision and two-component models are options of it.
  batch    many independent periodic runs of uneven cubes advanced together, then the fields of each.
  monitor  the readouts between steps: global FP64 sums and the droplet count of a state.
  conv     one 3x3x3 layer of the surrogate network forward (plain, or decoder input skip + upsampled).
  grad     the two gradients of such a layer (input gradient with flipped weights, weight gradient).
  predict  one surrogate jump from a handle's state: fields, network, candidate.
  train    one training step of the network up to its gradients: pack, forward, loss, backward.

Initial phase fields are emulsions of rounded power-diagram cells with smooth interfaces, made from
the seed on the GPU.  Boxes are nx x ny x nz with x fastest; walls bit 0, 1, 2 = x, y, z.
"""
import ctypes
import math
import os
import tempfile

import numpy as np
import torch

DEV = "cuda"
MASK5 = 0b11111  # phi, rho, ux, uy, uz
BYTES = {"twoset_f32": 432, "reduced_f32": 248, "reduced_f16": 140, "twoset_f64": 864, "moment_f32": 112}
SWEEP = (48, 64, 96, 128)
S_RHO, S_U, CH = 100.0, 100.0, 16  # scales and packed channels of the network's input and target


# ---------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------
def _lb(name, nx, ny, nz, steps, storage="twoset_f32", **o):
    c = dict(kind="lb", nx=nx, ny=ny, nz=nz, walls=0, steps=steps, storage=storage, tau_a=1.0, tau_b=1.0, A_h=0.0,
             h_min=3.0, h_max=3.0, g=0.0, g_mode=0, collision=0, model=0, fill="cells", film=8.0, tile=-1)
    c.update(o)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a single static droplet (Laplace checks, parameter studies): launches and latency count
        _lb("droplet_32", 32, 32, 32, 48, fill="one"),
        # two droplets driven at each other, the coalescence study of the near-contact force
        _lb("pair_64x64x128", 64, 64, 128, 12, fill="pair", A_h=0.1, g=1e-5, g_mode=2),
        # the headline run: dense emulsion in a channel, FP32 two-set, the tile that timing all of them picks
        _lb("emulsion_256x256x512", 256, 256, 512, 4, walls=2, A_h=0.1, g=1e-6, g_mode=1, tile=5),
        # a ragged channel with a viscosity ratio, the h^-3 tail and the regularised collision, exact reduced storage
        _lb("ragged_150x93x203", 150, 93, 203, 12, "reduced_f32", walls=2, A_h=0.08, h_min=2.0, h_max=5.0, tau_a=0.7,
            g=1e-6, g_mode=1, collision=1),
        # the emulsion in FP16-deviation storage, at the box the surrogate's trajectories use
        _lb("emulsion_f16_128x128x256", 128, 128, 256, 8, "reduced_f16", walls=2, A_h=0.1, g=1e-6, g_mode=1),
        # the Shan-Chen model of the same box
        _lb("shan_chen_128x128x256", 128, 128, 256, 8, walls=2, model=1, g=1e-6, g_mode=1),
        # the parameter sweep: 64 independent runs of 48^3 to 128^3
        dict(name="sweep_64_runs", kind="batch", runs=64, lo=48, hi=128, steps=12, storage="twoset_f32"),
        # drift monitors between steps
        dict(name="monitor_128x128x256", kind="monitor", nx=128, ny=128, nz=256, walls=2),
        # a decoder layer of the network at full resolution
        dict(name="conv_upcat_128x128x256", kind="conv", nx=128, ny=128, nz=256, cs=32, cl=64, cout=32),
        # a layer's gradients in training, one level down
        dict(name="grad_64x64x128", kind="grad", nx=64, ny=64, nz=128, cin=64, cout=64),
        # one surrogate jump of the trajectories' box
        dict(name="predict_128x128x256", kind="predict", nx=128, ny=128, nz=256),
        # one training step, half that box
        dict(name="train_128x128x128", kind="train", nx=128, ny=128, nz=128),
    ]


def _logint(rng, lo, hi, mult=1):
    return max(lo, min(hi, mult * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / mult)))


def draw(rng):
    kind = rng.choice(["lb", "lb", "lb", "lb", "batch", "monitor", "conv", "grad", "predict", "train"])
    if kind == "lb":
        nx, ny, nz = (_logint(rng, 24, m) for m in (256, 256, 512))
        model = rng.choice([0, 0, 0, 0, 1])
        storage = rng.choice(["twoset_f32", "twoset_f64"] if model else
                             ["twoset_f32", "twoset_f32", "reduced_f32", "reduced_f16", "moment_f32", "twoset_f64"])
        h_max = rng.choice([3.0, 3.0, 2.0, 4.5, 6.0])
        tau = rng.choice([1.0, 0.7, 0.9])
        return _lb(None, nx, ny, nz, rng.choice([2, 4] if nx * ny * nz > 4000000 else [4, 13, 27]), storage,
                   walls=rng.choice([0, 2, 2, 3, 6]), A_h=0.0 if model else rng.choice([0.0, 0.05, 0.1]),
                   h_min=min(h_max, 3.0), h_max=h_max, tau_a=tau, tau_b=rng.choice([1.0, tau]),
                   g=rng.choice([1e-6, 1e-5]), g_mode=rng.choice([0, 1, 2]), model=model,
                   collision=1 if storage == "moment_f32" else 0 if model else rng.choice([0, 0, 1]),
                   tile=rng.choice([-1, -1, -1, 1, 2, 3, 4, 5]))
    if kind == "batch":
        lo = rng.choice([24, 40, 48])
        return dict(kind="batch", runs=rng.randint(2, 40), lo=lo, hi=rng.choice([64, 96, 112]), steps=rng.choice([4, 14]),
                    storage=rng.choice(["twoset_f32", "reduced_f32", "reduced_f16"]))
    if kind == "monitor":
        nx, ny, nz = (_logint(rng, 24, m) for m in (256, 256, 400))
        return dict(kind="monitor", nx=nx, ny=ny, nz=nz, walls=rng.choice([0, 2]))
    if kind == "conv":
        nx, ny, nz = _logint(rng, 16, 128, 8), _logint(rng, 16, 128, 16), _logint(rng, 16, 256, 8)
        cl = rng.choice([0, 0, 2])
        cs = rng.choice([16, 32, 64, 128] if not cl else [32, 64])
        cout = rng.choice([32, 64, 128]) if not cl else cs
        while nx * ny * nz * cs * cout > 128 * 128 * 256 * 32 * 48:
            nz = max(16, nz // 16 * 8)
            nx = max(16, nx // 16 * 8)
            ny = max(16, ny // 32 * 16)
            if nx == ny == nz == 16:
                break
        if not cl and rng.random() < 0.4:  # extents off the tiled grid
            nx, ny, nz = (max(8, min(48, e) - rng.randint(0, 7)) for e in (nx, ny, nz))
        return dict(kind="conv", nx=nx, ny=ny, nz=nz, cs=cs, cl=cl * cs, cout=cout)
    if kind == "grad":
        nx, ny, nz = _logint(rng, 16, 96, 8), _logint(rng, 16, 96, 16), _logint(rng, 16, 96, 8)
        if rng.random() < 0.3:
            nx, ny, nz = (max(8, min(32, e) - rng.randint(0, 7)) for e in (nx, ny, nz))
        return dict(kind="grad", nx=nx, ny=ny, nz=nz, cin=rng.choice([32, 64, 96]), cout=rng.choice([32, 64]))
    nx, ny, nz = (8 * _logint(rng, 3, m) for m in (14, 14, 20))
    return dict(kind=kind, nx=nx, ny=ny, nz=nz)


# ---------------------------------------------------------------------------------------------
# inputs from the seed
# ---------------------------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _cells_phi(nx, ny, nz, walls, seed, film=8.0, width=1.3, spacing=26.0, keep=1.0):
    """phi [nz][ny][nx]: power-diagram cells of a jittered grid of seeds with weights r^2, r in [8, 12], rounded by a
    sphere and eroded by half a film, a tanh profile across each interface; `keep`: share of cells that hold a droplet."""
    g = np.random.default_rng(seed)
    n = np.array([nx, ny, nz])
    m = np.maximum(1, np.round(n / spacing)).astype(int)
    w = n / m
    cen = (np.stack(np.meshgrid(*[np.arange(k) for k in m], indexing="ij"), -1) + 0.5 +
           g.uniform(-0.2, 0.2, tuple(m) + (3,))) * w
    r2 = g.uniform(8.0, 12.0, tuple(m)) ** 2 * min(1.0, float(w.min()) / spacing) ** 2
    on = g.uniform(size=tuple(m)) <= keep
    on.flat[int(g.integers(on.size))] = True
    cen, r2, on = (torch.tensor(a, device=DEV, dtype=torch.float32) for a in (cen, r2, on.astype(np.float32)))
    z, y, x = torch.meshgrid(*[torch.arange(k, device=DEV, dtype=torch.float32) for k in (nz, ny, nx)], indexing="ij")
    pos = (x, y, z)
    cid = [torch.clamp((p / float(w[a])).long(), max=int(m[a]) - 1) for a, p in enumerate(pos)]

    def candidate(o):
        idx, ok = [], None
        for a in range(3):
            i = cid[a] + o[a]
            if (walls >> a) & 1:
                inside = (i >= 0) & (i < int(m[a]))
                ok = inside if ok is None else ok & inside
                i = i.clamp(0, int(m[a]) - 1)
            idx.append(i % int(m[a]))
        c = cen[idx[0], idx[1], idx[2]]
        d = []
        for a in range(3):
            e = pos[a] - c[..., a]
            d.append(e if (walls >> a) & 1 else e - float(n[a]) * torch.round(e / float(n[a])))
        p = d[0] ** 2 + d[1] ** 2 + d[2] ** 2 - r2[idx[0], idx[1], idx[2]]
        return p if ok is None else torch.where(ok, p, torch.full_like(p, 1e9)), idx, d

    offs = [(a, b, c) for c in (-1, 0, 1) for b in (-1, 0, 1) for a in (-1, 0, 1)]
    best, own, od = None, None, None
    for o in offs:
        p, idx, d = candidate(o)
        key = (idx[0] * int(m[1]) + idx[1]) * int(m[2]) + idx[2]
        if best is None:
            best, own, od = p, key, d
        else:
            t = p < best
            best, own = torch.where(t, p, best), torch.where(t, key, own)
            od = [torch.where(t, u, v) for u, v in zip(d, od)]
    margin = 0.5 * float(w.min()) - torch.sqrt(od[0] ** 2 + od[1] ** 2 + od[2] ** 2) + 0.15 * float(w.min())
    for o in offs:
        p, idx, d = candidate(o)
        key = (idx[0] * int(m[1]) + idx[1]) * int(m[2]) + idx[2]
        sep = torch.sqrt(sum((u - v) ** 2 for u, v in zip(d, od)))
        t = (p - best) / (2.0 * sep.clamp(min=1e-3))
        margin = torch.where(key == own, margin, torch.minimum(margin, t))
    for a in range(3):
        if (walls >> a) & 1:
            margin = torch.minimum(margin, torch.minimum(pos[a] - 0.5, float(n[a]) - 1.5 - pos[a]))
    phi = torch.tanh((margin - 0.5 * film) / width)
    return torch.where(on.reshape(-1)[own] > 0, phi, torch.full_like(phi, -1.0)).contiguous()


def _droplets(case, seed):
    """Centres and radii of the small cases' droplets."""
    r = np.random.default_rng(seed)
    n = np.array([case["nx"], case["ny"], case["nz"]], dtype=np.float64)
    if case["fill"] == "one":
        return (n / 2 + r.uniform(-1, 1, 3))[None, :], np.array([0.25 * n.min() + r.uniform(-0.5, 0.5)])
    c = n / 2 + r.uniform(-1.5, 1.5, (2, 3))
    c[0, 2], c[1, 2] = n[2] / 2 - 12.0 + r.uniform(-0.5, 0.5), n[2] / 2 + 12.0 + r.uniform(-0.5, 0.5)
    return c, 10.0 + r.uniform(-0.4, 0.4, 2)


def _flow(nx, ny, nz, seed):
    """rho and u [3] of a gentle flow: a few periodic modes."""
    r = np.random.default_rng(seed + 77)
    ax = [torch.arange(k, device=DEV, dtype=torch.float32) * (2 * math.pi / k) for k in (nx, ny, nz)]

    def mode(amp):
        k, p = r.integers(1, 3, 3), r.uniform(0, 2 * math.pi, 3)
        f = [torch.sin(int(k[a]) * ax[a] + float(p[a])) for a in range(3)]
        return amp * f[2][:, None, None] * f[1][None, :, None] * f[0][None, None, :]

    return (1.0 + mode(5e-3) + mode(5e-3)).contiguous(), torch.stack([mode(0.01) + mode(0.01) for _ in range(3)])


def _fields_of(case, seed):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    phi = _cells_phi(nx, ny, nz, case.get("walls", 2), seed, film=case.get("film", 8.0))
    return (phi,) + _flow(nx, ny, nz, seed)


def _lb_params(case):
    return dict(tau_a=case["tau_a"], tau_b=case["tau_b"], A_a=0.01, A_b=0.01, beta=0.7, A_h=case["A_h"],
                h_min=case["h_min"], h_max=case["h_max"], phi_I=0.9, g=(0.0, 0.0, case["g"]), g_mode=case["g_mode"],
                collision=case["collision"], model=case["model"], G=7.5 if case["model"] else 0.0, psi0=1.0)


def _sides(case):
    """Cube sides of a sweep's runs: the same for every seed."""
    allowed = [s for s in sorted(set(SWEEP) | {case["lo"], case["hi"]}) if case["lo"] <= s <= case["hi"]]
    return [int(s) for s in np.random.default_rng(2024 + case["runs"]).choice(allowed, case["runs"])]


def _sweep(case, seed):
    """(side, params, phi) of each run."""
    r = np.random.default_rng(seed)
    runs = []
    for side in _sides(case):
        A, Ah = float(r.uniform(0.005, 0.02)), float(r.uniform(0.05, 0.2))
        cells = max(1, round(side / 26.0)) ** 3
        p = dict(tau_a=1.0, tau_b=1.0, A_a=A, A_b=A, beta=0.7, A_h=Ah, h_min=3.0, h_max=3.0, phi_I=0.9,
                 g=(0.0, 0.0, 0.0), g_mode=0)
        phi = _cells_phi(side, side, side, 0, int(r.integers(1 << 30)), keep=min(1.0, int(r.integers(1, 21)) / cells))
        runs.append((side, p, phi))
    return runs


def _randn(shape, g, std=1.0):
    return torch.randn(shape, generator=g, device=DEV) * std


def _layer_table(base=32):
    c1, c2, c3, c4 = base, 2 * base, 4 * base, 8 * base
    return [("c1a", CH, c1), ("c1b", c1, c1), ("c2a", c1, c2), ("c2b", c2, c2), ("c3a", c2, c3), ("c3b", c3, c3),
            ("c4a", c3, c4), ("c4b", c4, c4), ("c5a", c3 + c4, c3), ("c5b", c3, c3), ("c6a", c2 + c3, c2),
            ("c6b", c2, c2), ("c7a", c1 + c2, c1), ("c7b", c1, c1), ("head", c1, CH)]


def _weights(seed):
    g, out = torch.Generator().manual_seed(int(seed)), {}
    for name, ci, co in _layer_table():
        taps = 1 if name == "head" else 27
        std = math.sqrt(2.0 / (taps * ci)) * (0.1 if name == "head" else 1.0)
        out[name] = ((torch.randn((co, taps, ci), generator=g) * std).numpy(), (torch.randn(co, generator=g) * 0.01).numpy())
    return out


# ---------------------------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------------------------
def prepare(case, seed):
    from paper_2405_14551_gb300 import lbcg as L
    kind = case["kind"]
    if kind == "lb":
        sim = L.Sim(case["nx"], case["ny"], case["nz"], walls=case["walls"], storage=case["storage"], **_lb_params(case))
        if case["tile"] >= 0:
            L.lb_set_tile(sim.h, case["tile"])
        if case["fill"] == "cells":
            sim.init_fields(*_fields_of(case, seed))
        else:
            sim.init_droplets(*_droplets(case, seed), width=1.3)
        return dict(kind=kind, sim=sim, steps=case["steps"])
    if kind == "batch":
        from paper_2405_14551_gb300 import workloads as W
        runs = [W.Workload("run", (s, s, s), 0, p, case["steps"], phi=phi) for s, p, phi in _sweep(case, seed)]
        b = L.Batch(runs, storage=case["storage"])
        L.lb_batch_set_tile(b.b, 5, 4)  # the shape the autotuner keeps for the sweep
        h = [b.run(r) for r in range(len(runs))]
        return dict(kind=kind, batch=b, h=h, steps=case["steps"], n=[w.shape[0] for w in runs], keep=runs)
    if kind == "monitor":
        sim = L.Sim(case["nx"], case["ny"], case["nz"], walls=case["walls"], A_h=0.1)
        sim.init_fields(*_fields_of(case, seed))
        return dict(kind=kind, sim=sim)
    if kind in ("conv", "grad"):
        g, bf = _gen(seed), torch.bfloat16
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        nv = nx * ny * nz
        s = dict(kind=kind, dims=(nx, ny, nz), status=torch.zeros(4, dtype=torch.int32, device=DEV), lib=L.load_library(),
                 check=L._check, stream=ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if kind == "conv":
            cin, cout = case["cs"] + case["cl"], case["cout"]
            s["x"] = _randn((nv, case["cs"]), g).relu().to(bf)
            if case["cl"]:
                s["low"] = _randn((nv // 8, case["cl"]), g).relu().to(bf)
            s["w"] = _randn((cout, 27, cin), g, math.sqrt(2.0 / (27 * cin))).to(bf)
            s["b"] = _randn((cout,), g, 0.1)
            s["y"] = torch.empty((nv, cout), dtype=bf, device=DEV)
        else:
            cin, cout = case["cin"], case["cout"]
            s["x"] = _randn((nv, cin), g).relu().to(bf)
            s["dy"] = _randn((nv, cout), g, 1e-3).to(bf)
            s["w"] = _randn((cout, 27, cin), g, math.sqrt(2.0 / (27 * cin))).to(bf)
            s["wt"] = torch.empty((cin, 27, cout), dtype=bf, device=DEV)
            s["dx"] = torch.empty((nv, cin), dtype=torch.float32, device=DEV)
            s["dw"] = torch.empty((cout, 27, cin), dtype=torch.float32, device=DEV)
        return s
    from paper_2405_14551_gb300 import surrogate as S
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    net = S.UNet(base=32)
    net.load_parameters(_weights(seed))
    phi, rho, u = _fields_of(case, seed)
    if kind == "predict":
        sim = L.Sim(nx, ny, nz, walls=2, **S.workload_params())
        fd, path = tempfile.mkstemp(suffix=".lbnn")
        os.close(fd)
        try:
            net.save(path)
            L.lb_surrogate_load(sim.h, path)
        finally:
            os.remove(path)
        sim.init_fields(phi, rho, u)
        return dict(kind=kind, sim=sim, out=torch.empty((5, nz, ny, nx), dtype=torch.float32, device=DEV))
    f0, f1 = _pair(phi, rho, u)
    n = nx * ny * nz
    w = torch.zeros(CH, dtype=torch.float32, device=DEV)
    w[:5] = torch.tensor([4.0, 1.0, 1.0, 1.0, 1.0])
    return dict(kind=kind, net=net, f0=f0, f1=f1, shape=(nx, ny, nz, 1), wch=w, stream=torch.cuda.current_stream(),
                x=torch.empty((n, CH), dtype=torch.bfloat16, device=DEV), t=torch.empty((n, CH), device=DEV),
                g=torch.empty((n, CH), device=DEV), loss=torch.zeros(1, dtype=torch.float64, device=DEV))


def _pair(phi, rho, u):
    """Two snapshots [5][N] for training: the second shifted by the flow along z."""
    f0 = torch.cat([phi[None], rho[None], u]).reshape(5, -1).contiguous()
    f1 = torch.cat([torch.roll(v, 1, 0)[None] for v in (phi, rho, *u)]).reshape(5, -1).contiguous()
    return f0, f1


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def run(state):
    from paper_2405_14551_gb300 import lbcg as L
    s, kind = state, state["kind"]
    if kind == "lb":
        s["sim"].step(s["steps"])
        return {"fields": s["sim"].fields_device(MASK5)}
    if kind == "batch":
        s["batch"].step(s["steps"])
        out = []
        for h, n in zip(s["h"], s["n"]):
            out.append(torch.empty((5, n, n, n), dtype=torch.float32, device=DEV))
            L.lb_fields(h, MASK5, out[-1], True)
        return out
    if kind == "monitor":
        return {"sums": s["sim"].reduce(), "droplets": s["sim"].droplet_count()}
    nx, ny, nz = s["dims"] if "dims" in s else (0, 0, 0)
    if kind == "conv":
        cout = s["w"].shape[0]
        if "low" in s:
            s["check"](s["lib"].lbnn_conv3d_fwd_upcat(
                _ptr(s["x"]), s["x"].shape[1], _ptr(s["low"]), s["low"].shape[1], _ptr(s["w"]), _ptr(s["b"]), _ptr(s["y"]),
                None, cout, 0, nx, ny, nz, 1, 5, 1, _ptr(s["status"]), s["stream"]), "conv")
        else:
            s["check"](s["lib"].lbnn_conv3d_fwd(
                _ptr(s["x"]), s["x"].shape[1], _ptr(s["w"]), 27, _ptr(s["b"]), _ptr(s["y"]), None, cout, 0, nx, ny, nz, 1,
                5, 1, _ptr(s["status"]), s["stream"]), "conv")
        return {"y": s["y"]}
    if kind == "grad":
        cout, _, cin = s["w"].shape
        s["dw"].zero_()
        s["check"](s["lib"].lbnn_conv3d_wgrad(_ptr(s["dy"]), cout, _ptr(s["x"]), cin, 27, _ptr(s["dw"]), nx, ny, nz, 1, 5,
                                              4096, _ptr(s["status"]), s["stream"]), "wgrad")
        s["check"](s["lib"].lbnn_flip_weights(_ptr(s["w"]), cout, 27, cin, _ptr(s["wt"]), s["stream"]), "flip")
        s["check"](s["lib"].lbnn_conv3d_fwd(_ptr(s["dy"]), cout, _ptr(s["wt"]), 27, None, None, _ptr(s["dx"]), cin, 0, nx,
                                            ny, nz, 1, 5, 0, _ptr(s["status"]), s["stream"]), "dgrad")
        return {"dw": s["dw"], "dx": s["dx"]}
    if kind == "predict":
        L.lb_surrogate_predict(s["sim"].h, s["out"])
        return {"candidate": s["out"]}
    from paper_2405_14551_gb300 import surrogate as S
    net = s["net"]
    S.pack_input(s["f0"], s["x"], s["stream"])
    S.pack_target(s["f0"], s["f1"], s["t"], s["stream"])
    y = net.forward(s["x"], s["shape"])
    s["loss"].zero_()
    S.mse(y, s["t"], s["wch"], s["g"], s["loss"], s["stream"])
    net.backward(s["g"])
    return {"loss": s["loss"].float(), "y": y, "gw": dict(net.gw), "gb": dict(net.gb)}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        n = float(sum(s**3 for s in _sides(case)))
        return {"bytes": n * (case["steps"] * BYTES[case["storage"]] + 20), "flops": n * case["steps"] * 900.0}
    n = float(case["nx"]) * case["ny"] * case["nz"]
    if kind == "lb":
        return {"bytes": n * (case["steps"] * BYTES[case["storage"]] + 20), "flops": n * case["steps"] * 900.0}
    if kind == "monitor":
        return {"bytes": 20.0 * n, "flops": 200.0 * n}
    if kind == "conv":
        cin, cout = case["cs"] + case["cl"], case["cout"]
        return {"bytes": 2 * n * (case["cs"] + case["cl"] / 8 + cout) + 54 * cin * cout, "flops": 54 * n * cin * cout}
    if kind == "grad":
        cin, cout = case["cin"], case["cout"]
        return {"bytes": 2 * n * (cin + cout) + 4 * n * cin + 162 * cin * cout, "flops": 108 * n * cin * cout}
    f = sum((2 if name == "head" else 54) * n * ci * co / 8 ** {"1": 0, "7": 0, "h": 0, "2": 1, "6": 1, "3": 2, "5": 2,
                                                                "4": 3}[name[1] if name != "head" else "h"]
            for name, ci, co in _layer_table())
    if kind == "predict":
        return {"bytes": 40 * n, "flops": f}
    return {"bytes": 40 * n + 64 * n, "flops": 3 * f}


# ---------------------------------------------------------------------------------------------
# the same results in 64 bits, from the formulas
# ---------------------------------------------------------------------------------------------
C27 = [(i % 3 - 1, i // 3 % 3 - 1, i // 9 - 1) for i in range(27)]
NORM2 = [sum(v * v for v in c) for c in C27]
W27 = [(8 / 27, 2 / 27, 1 / 54, 1 / 216)[k] for k in NORM2]


def _at(a, c):
    """a(x + c) with periodic wrap, a [..., nz, ny, nx]."""
    return torch.roll(a, (-c[2], -c[1], -c[0]), (-3, -2, -1)) if any(c) else a


def _grad3(a, solid):
    g = [torch.zeros_like(a) for _ in range(3)]
    for c, w in zip(C27, W27):
        if not any(c):
            continue
        v = _at(a, c)
        if solid is not None:
            v = torch.where(_at(solid, c), a, v)
        for k in range(3):
            if c[k]:
                g[k] += (3 * w * c[k]) * v
    return g


def _dot(c, v):
    s = 0.0
    for k in range(3):
        if c[k]:
            s = s + c[k] * v[k]
    return s


def _scan(phi, g, gg, solid, walls, P):
    """Distance h to a second interface along the outward normal, 0 where there is none."""
    nz, ny, nx = phi.shape
    dims, K = (nx, ny, nz), int(math.floor(P["h_max"]))
    fl = (phi.abs() < P["phi_I"]) & (gg >= 1e-2)
    if solid is not None:
        fl &= ~solid
    h = torch.zeros(phi.numel(), dtype=torch.float64, device=DEV)
    at = fl.reshape(-1).nonzero()[:, 0]
    pos = (at % nx, at // nx % ny, at // (nx * ny))
    gf, gn, pf = [v.reshape(-1) for v in g], gg.reshape(-1), phi.reshape(-1)
    no = [-v[at] / gn[at] for v in gf]
    open_ = torch.ones_like(at, dtype=torch.bool)
    for k in range(1, K + 1):
        q = [p + (torch.sign(v) * torch.floor((k * v).abs() + 0.5)).long() for p, v in zip(pos, no)]
        for a in range(3):
            if (walls >> a) & 1:
                open_ &= (q[a] > 0) & (q[a] < dims[a] - 1)
            q[a] = q[a] % dims[a]
        t = q[0] + nx * (q[1] + ny * q[2])
        d = sum(gf[a][at] * gf[a][t] for a in range(3))
        hit = open_ & (pf[t].abs() < P["phi_I"]) & (gn[t] >= 1e-2) & (d < -1e-6 * gn[at] * gn[t])
        h[at[hit]] = float(k)
        open_ &= ~hit
    return h.reshape(phi.shape)


def _force(phi, rho, rA, P, walls, solid):
    """(colour gradient, its norm, total force) at one level."""
    g = _grad3(phi, solid)
    gg = torch.sqrt(g[0] ** 2 + g[1] ** 2 + g[2] ** 2)
    F = [torch.zeros_like(phi) for _ in range(3)]
    if P["A_h"]:
        h = _scan(phi, g, gg, solid, walls, P)
        a = torch.where(h <= P["h_min"], torch.full_like(h, P["A_h"]), P["A_h"] * (P["h_min"] / h.clamp(min=1)) ** 3)
        a = torch.where((h > 0) & (h <= P["h_max"]), a, torch.zeros_like(a))
        F = [0.5 * a * v for v in g]
    return g, gg, _body(F, rho, rA, P)


def _body(F, rho, rA, P):
    if P["g_mode"] == 1:
        F[2] = F[2] + rho * P["g"][2]
    elif P["g_mode"] == 2:
        z = torch.arange(rho.shape[0], device=DEV)[:, None, None]
        s = torch.where((z == 0) | (2 * z == rho.shape[0]), 0.0, torch.where(2 * z < rho.shape[0], 1.0, -1.0)).double()
        F[2] = F[2] + s * rA * P["g"][2]
    return F


def _psi_force(rA, rB, P, solid):
    pa, pb = (P["psi0"] * (1 - torch.exp(-r / P["psi0"])) for r in (rA, rB))
    ga, gb = _grad3(pa, solid), _grad3(pb, solid)
    FA, FB = [-pa * P["G"] / 3 * v for v in gb], [-pb * P["G"] / 3 * v for v in ga]
    if P["g_mode"] == 1:
        FA[2], FB[2] = FA[2] + rA * P["g"][2], FB[2] + rB * P["g"][2]
    else:
        FA = _body(FA, rA, rA, P)
    return FA, FB


def _moments(f):
    rho = f.sum(0)
    j = [torch.zeros_like(rho) for _ in range(3)]
    for i, c in enumerate(C27):
        for k in range(3):
            if c[k]:
                j[k] += c[k] * f[i]
    return rho, j


def _exact_lb(phi, rho, u, walls, P, model, collision, steps):
    """Fields [5][nz][ny][nx] after `steps` steps from component equilibria, in 64 bits."""
    phi, rho, u = phi.double(), rho.double(), u.double()
    nz, ny, nx = phi.shape
    solid = None
    if walls:
        solid = torch.zeros(phi.shape, dtype=torch.bool, device=DEV)
        for a, dim in ((0, 2), (1, 1), (2, 0)):
            if (walls >> a) & 1:
                solid.select(dim, 0).fill_(True)
                solid.select(dim, phi.shape[dim] - 1).fill_(True)
    uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
    fA, fB = (torch.empty((27,) + phi.shape, dtype=torch.float64, device=DEV) for _ in range(2))
    for i, c in enumerate(C27):
        cu = _dot(c, u)
        fe = W27[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)
        fA[i] = 0.5 * (1 + phi) * fe
        fB[i] = fe - fA[i]
    first = phi
    for t in range(steps + 1):
        rA, rB = fA.sum(0), fB.sum(0)
        if solid is not None:
            rA, rB = (torch.where(solid, torch.full_like(r, 0.5), r) for r in (rA, rB))
        phi = first if t == 0 else (rA - rB) / (rA + rB)
        rho = rA + rB
        if model:
            (_, jA), (_, jB) = _moments(fA), _moments(fB)
            FA, FB = _psi_force(rA, rB, P, solid)
            F = [a + b for a, b in zip(FA, FB)]
            j = [a + b for a, b in zip(jA, jB)]
        else:
            j = _moments(fA + fB)[1]
            g, gg, F = _force(phi, rho, rA, P, walls, solid)
        u = [(j[k] + 0.5 * F[k]) / rho for k in range(3)]
        if t == steps:
            out = torch.stack([phi, rho, *u])
            return out if solid is None else torch.where(solid, torch.zeros_like(out), out)
        if model:
            wa, wb = 1 / P["tau_a"], 1 / P["tau_b"]
            v = [(wa * (jA[k] + 0.5 * FA[k]) + wb * (jB[k] + 0.5 * FB[k])) / (wa * rA + wb * rB) for k in range(3)]
            vv = v[0] ** 2 + v[1] ** 2 + v[2] ** 2
            for i, c in enumerate(C27):
                cu = _dot(c, v)
                e = W27[i] * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * vv)
                for f, r, w, Fk in ((fA, rA, wa, FA), (fB, rB, wb, FB)):
                    S = (1 - 0.5 * w) * W27[i] * sum((3 * (c[k] - v[k]) + 9 * cu * c[k]) * Fk[k] for k in range(3))
                    f[i] += w * (r * e - f[i]) + S
        else:
            f = fA.add_(fB)
            ta, tb = P["tau_a"], P["tau_b"]
            tau = 0.5 + 3 / ((rA / rho) / ((ta - 0.5) / 3) + (rB / rho) / ((tb - 0.5) / 3)) if ta != tb else ta
            om = 1 / tau
            uu, uF = u[0] ** 2 + u[1] ** 2 + u[2] ** 2, sum(u[k] * F[k] for k in range(3))
            seg, sA = 0.7 * rA * rB / rho / gg.clamp(min=1e-4), rA / rho
            A2 = 0.5 * (P["A_a"] + P["A_b"])
            inv = torch.where(gg >= 1e-12, 1 / gg.clamp(min=1e-300), torch.zeros_like(gg))
            if collision:
                pi = {}
                for a in range(3):
                    for b in range(a, 3):
                        pi[a, b] = sum(c[a] * c[b] * f[i] for i, c in enumerate(C27) if c[a] * c[b]) - rho * (
                            u[a] * u[b] + (1 / 3 if a == b else 0))
                tr = pi[0, 0] + pi[1, 1] + pi[2, 2]
            for i, c in enumerate(C27):
                w, cu, cF, cg = W27[i], _dot(c, u), _dot(c, F), _dot(c, g)
                fe = w * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)
                if collision:
                    q = sum((1 if a == b else 2) * c[a] * c[b] * pi[a, b] for a, b in pi if c[a] * c[b])
                    fs = fe + (1 - om) * w * (-1.5 * cF + 4.5 * (q - tr / 3))
                else:
                    fs = (1 - om) * f[i] + om * fe
                fs = fs + A2 * (w * cg * cg * inv - gg * w * (NORM2[i] - 2 / 3))
                fs = fs + (1 - 0.5 * om) * w * (3 * (cF - uF) + 9 * cu * cF)
                fA[i] = sA * fs + seg * w * cg * (NORM2[i] ** -0.5 if NORM2[i] else 0.0)
                fB[i] = fs - fA[i]
        for f in (fA, fB):  # stream: pull from x - c, or bounce back
            if solid is None:
                for i, c in enumerate(C27):
                    if any(c):
                        f[i] = _at(f[i], tuple(-k for k in c))
            else:
                for i in range(13):
                    c, o = C27[i], 26 - i
                    back = tuple(-k for k in c)
                    fi = torch.where(_at(solid, back), f[o], _at(f[i], back))
                    f[o] = torch.where(_at(solid, c), f[i], _at(f[o], c))
                    f[i] = fi
    raise AssertionError


def _tap(x, t, fill=None):
    """x(v + offset of tap t) of x [nz][ny][nx][c]: periodic in x and z, zero beyond y."""
    c = C27[t]
    v = torch.roll(x, (-c[2], -c[1], -c[0]), (0, 1, 2)) if any(c) else x
    if c[1]:
        v = v.clone()
        v[:, -1 if c[1] > 0 else 0] = 0
    return v


class _Conv(torch.autograd.Function):
    """3x3x3 convolution by 27 matrix products, w [co][27][ci]; gradients the same way."""

    @staticmethod
    def forward(ctx, x, w):
        ctx.save_for_backward(x, w)
        y = None
        for t in range(27):
            p = _tap(x, t) @ w[:, t].T
            y = p if y is None else y.add_(p)
        return y

    @staticmethod
    def backward(ctx, gy):
        x, w = ctx.saved_tensors
        gx, gw = torch.zeros_like(x), torch.empty_like(w)
        flat = gy.reshape(-1, gy.shape[-1])
        for t in range(27):
            gw[:, t] = flat.T @ _tap(x, t).reshape(-1, x.shape[-1])
            gx += _tap(gy, 26 - t) @ w[:, t]
        return gx, gw


def _up(x):
    return x.repeat_interleave(2, 0).repeat_interleave(2, 1).repeat_interleave(2, 2)


def _pool(x):
    z, y, xx, c = x.shape
    return x.reshape(z // 2, 2, y // 2, 2, xx // 2, 2, c).mean((1, 3, 5))


def _exact_net(x, p):
    def conv(name, v):
        return torch.relu(_Conv.apply(v, p[name][0]) + p[name][1])

    s1 = conv("c1b", conv("c1a", x))
    s2 = conv("c2b", conv("c2a", _pool(s1)))
    s3 = conv("c3b", conv("c3a", _pool(s2)))
    b4 = conv("c4b", conv("c4a", _pool(s3)))
    d3 = conv("c5b", conv("c5a", torch.cat([s3, _up(b4)], -1)))
    d2 = conv("c6b", conv("c6a", torch.cat([s2, _up(d3)], -1)))
    d1 = conv("c7b", conv("c7a", torch.cat([s1, _up(d2)], -1)))
    return d1 @ p["head"][0][:, 0].T + p["head"][1]


def _exact_params(seed):
    return {k: (torch.tensor(w, device=DEV).bfloat16().double(), torch.tensor(b, device=DEV).double())
            for k, (w, b) in _weights(seed).items()}


def _net_input(f):
    s = torch.zeros(f.shape[1:] + (CH,), dtype=torch.float64, device=DEV)
    for k, (a, b) in enumerate(((0, 1), (1, S_RHO), (0, S_U), (0, S_U), (0, S_U))):
        s[..., k] = (b * (f[k].float() - a)).bfloat16().double()
    return s


@torch.no_grad()
def exact(case, seed):
    kind = case["kind"]
    if kind == "lb":
        if case["fill"] == "cells":
            phi, rho, u = _fields_of(case, seed)
        else:
            cen, rad = _droplets(case, seed)
            z, y, x = torch.meshgrid(*[torch.arange(case[k], device=DEV, dtype=torch.float64) for k in ("nz", "ny", "nx")],
                                     indexing="ij")
            phi = torch.full_like(x, -1.0)
            for c, r in zip(cen, rad):
                d = [v - float(c[a]) for a, v in enumerate((x, y, z))]
                d = [v - n * torch.round(v / n) for v, n in zip(d, (case["nx"], case["ny"], case["nz"]))]
                phi = torch.maximum(phi, torch.tanh((float(r) - torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)) / 1.3))
            phi = phi.float()
            rho, u = torch.ones_like(phi), torch.zeros((3,) + tuple(phi.shape), device=DEV)
        return {"fields": _exact_lb(phi, rho, u, case["walls"], _lb_params(case), case["model"], case["collision"],
                                    case["steps"])}
    if kind == "batch":
        return [_exact_lb(phi, torch.ones_like(phi), torch.zeros((3,) + tuple(phi.shape), device=DEV), 0, p, 0, 0,
                          case["steps"]) for _, p, phi in _sweep(case, seed)]
    if kind == "monitor":
        phi, rho, u = _fields_of(case, seed)
        P = dict(A_h=0.1, h_min=3.0, h_max=3.0, phi_I=0.9, A_a=0.01, A_b=0.01, tau_a=1.0, tau_b=1.0, g_mode=0)
        f = _exact_lb(phi, rho, u, case["walls"], P, 0, 0, 0)
        fl = f[1] > 0
        ph, r, v = f[0], f[1], f[2:]
        g, gg, _ = _force(phi.double(), rho.double(), rho.double(), dict(P, A_h=0.0), case["walls"], ~fl if case["walls"] else None)
        active = (_scan(phi.double(), g, gg, ~fl if case["walls"] else None, case["walls"], P) > 0).sum()
        s = torch.stack([(r * (1 + ph) / 2).sum(), (r * (1 - ph) / 2).sum(), *[(r * c).sum() for c in v],
                         ((1 + ph) / 2)[fl].sum(), active.double(), (0.5 * r * (v ** 2).sum(0)).sum()])
        return {"sums": s.cpu().numpy(), "droplets": None}
    if kind in ("conv", "grad"):
        s = prepare(case, seed)
        nx, ny, nz = s["dims"]
        x = s["x"].double().reshape(nz, ny, nx, -1)
        if kind == "conv":
            if "low" in s:
                x = torch.cat([x, _up(s["low"].double().reshape(nz // 2, ny // 2, nx // 2, -1))], -1)
            y = torch.relu(_Conv.apply(x, s["w"].double()) + s["b"].double())
            return {"y": y.reshape(nx * ny * nz, -1)}
        dy, w = s["dy"].double().reshape(nz, ny, nx, -1), s["w"].double()
        dx = _Conv.apply(dy, torch.flip(w, (1,)).permute(2, 1, 0).contiguous())
        flat = dy.reshape(-1, dy.shape[-1])
        dw = torch.stack([flat.T @ _tap(x, t).reshape(-1, x.shape[-1]) for t in range(27)], 1)
        return {"dw": dw, "dx": dx.reshape(nx * ny * nz, -1)}
    phi, rho, u = _fields_of(case, seed)
    p = _exact_params(seed)
    if kind == "predict":
        f = _exact_lb(phi, rho, u, 2, dict(A_h=0.1, h_min=3.0, h_max=3.0, phi_I=0.9, A_a=0.01, A_b=0.01, tau_a=1.0, tau_b=1.0,
                                           g_mode=1, g=(0.0, 0.0, 1e-6)), 0, 0, 0)
        y = _exact_net(_net_input(f), p)
        out = torch.stack([(f[0] + y[..., 0]).clamp(-1, 1), (f[1] + y[..., 1] / S_RHO).clamp(min=0.5),
                           *[f[k] + y[..., k] / S_U for k in (2, 3, 4)]])
        return {"candidate": out}
    f0, f1 = (f.reshape(5, case["nz"], case["ny"], case["nx"]) for f in _pair(phi, rho, u))
    t = torch.stack([f1[0] - f0[0], *[100.0 * (f1[k] - f0[k]) for k in (1, 2, 3, 4)]], -1).double()
    with torch.enable_grad():
        p = {k: (w.requires_grad_(), b.requires_grad_()) for k, (w, b) in p.items()}
        y = _exact_net(_net_input(f0), p)
        wch = torch.tensor([4.0, 1.0, 1.0, 1.0, 1.0], dtype=torch.float64, device=DEV)
        loss = (wch * (y[..., :5] - t) ** 2).sum() / (t.numel())
        loss.backward()
    return {"loss": loss.detach().reshape(1), "y": y.detach().reshape(-1, CH), "gw": {k: v[0].grad for k, v in p.items()},
            "gb": {k: v[1].grad for k, v in p.items()}}
