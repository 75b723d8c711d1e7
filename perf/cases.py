"""What a user of this framework has it do, as cases that can be timed: the solver (three models, two precision
forms, single grids and batches), the warm-start network (training step, inference, one wide layer) and the seed
constraint that follows it.

  listed()             the cases
  draw(rng)            one more of the same ranges
  prepare(case, seed)  what a program holds before the call: grids with geometry (their tiles tuned where the case
                       says so, as programs with long runs do), pinned host states, networks
  run(state)           one pass through the public entry points (pf.Grid, pf.Batch, nn.UNet, the C ABI)
  work(case)           bytes and operations the pass cannot do without
  exact(case, seed)    the same outputs from plain torch in binary64

Solver passes are whole calls: the state goes in from pinned host memory, the run is made on the device, the state
comes back to pinned host memory."""
import ctypes
import math

import numpy as np
import torch

from paper_2401_01672_gb300 import inputs as I
from paper_2401_01672_gb300 import nn as NN
from paper_2401_01672_gb300 import pf

MODELS = {"full": I.MODEL_FULL, "temp": I.MODEL_TEMP, "micro": I.MODEL_MICRO}
REACTIONS = {"sigmap1p": I.REACT_SIGMAP1P, "gradp": I.REACT_GRADP}
PRECISIONS = {"f64": I.PREC_FP64, "f32": I.PREC_FP32}
DEV = "cuda"


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest grid of the framework's configurations: the 32^3 micro-scale grain, 200 steps of a fixed
        # size; every kernel is short, so launches and the gaps between them count
        dict(name="micro_32_f64", kind="grid", model="micro", reaction="sigmap1p", prec="f64", n1=32, n2=32, n3=32,
             steps=200, adaptive=False, tuned=False),
        # the paper's macro-scale vessel at N3 = 100 (50 x 50 x 100 cells, glass cap, Dirichlet top): half a million
        # adaptive attempts a run in real use; the row of 50 cells is ragged against every tile
        dict(name="macro_100_f64", kind="vessel", model="full", reaction="sigmap1p", prec="f64", n3=100, steps=32,
             adaptive=True, tuned=True),
        # the same vessel in the temperature-focused model (a tanh and two blends per cell instead of a phase field)
        dict(name="macro_100_temp", kind="vessel", model="temp", reaction="sigmap1p", prec="f64", n3=100, steps=12,
             adaptive=True, tuned=True),
        # the vessel at N3 = 200 in the binary32-field form (the mesh-resolution study)
        dict(name="macro_200_f32", kind="vessel", model="full", reaction="sigmap1p", prec="f32", n3=200, steps=64,
             adaptive=False, tuned=True),
        # the headline workload: 256^3 bead packing, binary64, the freezing front at half height, adaptive steps
        dict(name="bead_256_f64", kind="grid", model="full", reaction="sigmap1p", prec="f64", n1=256, n2=256, n3=256,
             steps=12, adaptive=True, tuned=True),
        # a large bead packing in the binary32-field form (the form for long runs on large grids)
        dict(name="bead_320_f32", kind="grid", model="full", reaction="sigmap1p", prec="f32", n1=320, n2=320, n3=320,
             steps=64, adaptive=False, tuned=True),
        # the parametric sweep: micro-scale instances of uneven size, each with its own step, in one batch
        dict(name="sweep_12_f32", kind="batch", prec="f32", count=12, lo=96, hi=192, steps=16, tuned=True),
        # relaxation of one micro-scale instance in binary64 with the equilibrium test (the judge of a warm start)
        dict(name="relax_128_f64", kind="batch", prec="f64", count=1, lo=128, hi=128, steps=24, tuned=False),
        # one training step of the warm-start network at the default batch: four crops of 64^3, forward, backward, Adam
        dict(name="train_4x64", kind="train", batch=4, side=64),
        # inference on a 256^3 packing
        dict(name="infer_256", kind="infer", batch=1, side=256),
        # a wide layer of that inference by itself (first decoder convolution, 64^3 voxels, 128 -> 64 channels)
        dict(name="conv_64_128to64", kind="conv", n=1, side=64, cin=128, cout=64),
        # the prediction kept in the ice region connected to the seed, 256^3
        dict(name="seed_256", kind="seed", n1=256, n2=256, n3=256),
    ]


def draw(rng):
    def logint(lo, hi, step=1):
        v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)) * step
        return max(lo, min(hi, v))

    # (adaptive runs are short: at the stability limit the step sequence amplifies rounding about a decade every
    # four attempts, in the temperature-focused model most)
    kind = rng.choice(["grid", "grid", "grid", "vessel", "vessel", "batch", "batch", "train", "infer", "conv", "seed"])
    if kind == "grid":
        model, prec = rng.choice(["full", "full", "micro"]), rng.choice(["f64", "f32"])
        n = [logint(32, 256) for _ in range(3)]
        if rng.random() < 0.5:
            n = [8 * max(4, round(v / 8)) for v in n]
        adaptive = prec == "f64" and rng.random() < 0.7
        return dict(kind=kind, model=model, reaction=rng.choice(["sigmap1p", "sigmap1p", "gradp"]), prec=prec, n1=n[0],
                    n2=n[1], n3=n[2], steps=rng.choice([6, 8, 12] if adaptive else [8, 16, 24]), adaptive=adaptive,
                    tuned=rng.random() < 0.5)
    if kind == "vessel":
        model, prec = rng.choice(["full", "full", "temp"]), rng.choice(["f64", "f32"])
        return dict(kind=kind, model=model, reaction=rng.choice(["sigmap1p", "gradp"]) if model == "full" else "sigmap1p",
                    prec=prec, n3=logint(60, 240, 2), steps=rng.choice([8, 12] if prec == "f64" else [16, 32, 64]),
                    adaptive=prec == "f64", tuned=True)
    if kind == "batch":
        lo = logint(48, 128, 8)
        return dict(kind=kind, prec=rng.choice(["f32", "f32", "f64"]), count=rng.randint(1, 8), lo=lo,
                    hi=min(192, lo + 8 * rng.randint(0, 8)), steps=rng.choice([8, 16, 24]), tuned=rng.random() < 0.5)
    if kind == "train":
        side = rng.choice([32, 48, 64])
        return dict(kind=kind, batch=rng.randint(1, 8 if side < 64 else 4), side=side)
    if kind == "infer":
        return dict(kind=kind, batch=1, side=8 * rng.randint(6, 28))
    if kind == "conv":
        return dict(kind=kind, n=rng.randint(1, 4), side=logint(12, 64), cin=rng.choice([16, 32, 64, 128]),
                    cout=rng.choice([16, 32, 64, 128]))
    return dict(kind="seed", n1=logint(64, 256), n2=logint(64, 256), n3=logint(64, 256))


# ------------------------------------------------------------------ inputs
def packing(shape, solid, r_lo, r_hi, g):
    """Overlapping beads, radii uniform in [r_lo, r_hi] voxels, as many as give the solid fraction on average;
    rows (x, y, z, r) in voxels."""
    mean_vol = math.pi / 3.0 * (r_hi ** 4 - r_lo ** 4) / (r_hi - r_lo)
    n = max(1, round(-math.log(1.0 - solid) * shape[0] * shape[1] * shape[2] / mean_vol))
    c = g.uniform(0.0, 1.0, (n, 3)) * np.array(shape, dtype=np.float64)
    return np.hstack([c, g.uniform(r_lo, r_hi, (n, 1))])


def surface_distance(shape, spheres, reach):
    """Signed distance of every cell centre to the nearest bead surface (voxels, (n3, n2, n1)), +inf beyond `reach`."""
    n1, n2, n3 = shape
    d = torch.full((n3, n2, n1), math.inf, dtype=torch.float64, device=DEV)
    ax = [torch.arange(n, dtype=torch.float64, device=DEV) + 0.5 for n in shape]
    for x, y, z, r in spheres:
        lo = [max(0, math.floor(c - r - reach)) for c in (x, y, z)]
        hi = [min(n, math.ceil(c + r + reach) + 1) for c, n in zip((x, y, z), shape)]
        if any(a >= b for a, b in zip(lo, hi)):
            continue
        s = ((ax[2][lo[2]:hi[2]] - z) ** 2)[:, None, None] + ((ax[1][lo[1]:hi[1]] - y) ** 2)[:, None] + \
            (ax[0][lo[0]:hi[0]] - x) ** 2
        v = d[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]]
        torch.minimum(v, torch.sqrt(s) - r, out=v)
    return d


def glass(shape, h, spheres, xi_G, x3_cap):
    """The glass field of Sec. 2.1 from beads in metres, (n3, n2, n1); farther than 40 xi_G from every bead its tail is
    below 1e-17."""
    d = surface_distance(shape, spheres / h, 40.0 * xi_G / h)
    G = 0.5 * (1.0 - torch.tanh(d * (h / (2.0 * xi_G))))
    if not math.isnan(x3_cap):
        z = (torch.arange(shape[2], dtype=torch.float64, device=DEV) + 0.5) * h
        G = torch.maximum(G, 0.5 * (1.0 + torch.tanh((z - x3_cap) / (2.0 * xi_G)))[:, None, None])
    return G


def front_state(shape, h, xi, solid, front, cold, warm):
    """The freezing front at the fraction `front` of the height: phi the planar interface profile in the pores (0 in
    the glass), theta linear from the cold top to 0 at the front and up to `warm` twenty cells below it."""
    n1, n2, n3 = shape
    z = (torch.arange(n3, dtype=torch.float64, device=DEV) + 0.5) * h
    L, zf = n3 * h, front * n3 * h
    prof = 0.5 * (1.0 + torch.tanh((z - zf) / (2.0 * xi)))
    th = torch.where(z >= zf, cold * (z - zf) / (L - zf), warm * torch.clamp((zf - z) / (20 * h), max=1.0))
    phi = torch.where(solid, torch.zeros((), dtype=torch.float64, device=DEV), prof[:, None, None])
    return th[:, None, None].expand(n3, n2, n1).contiguous(), phi.contiguous()


def ball_state(shape, center, radius, xi, solid):
    """An ice grain of `radius` voxels with its interface profile, in the pores."""
    n1, n2, n3 = shape
    ax = [torch.arange(n, dtype=torch.float64, device=DEV) + 0.5 - c for n, c in zip(shape, center)]
    r = torch.sqrt((ax[2] ** 2)[:, None, None] + (ax[1] ** 2)[:, None] + ax[0] ** 2)
    phi = 0.5 * (1.0 - torch.tanh((r - radius) / (2.0 * xi)))
    return torch.where(solid, torch.zeros_like(phi), phi)


def pinned(t):
    out = torch.empty(t.numel(), dtype=t.dtype, pin_memory=True)
    out.copy_(t.reshape(-1))
    return out


def problem(case, seed):
    """One grid's problem: sizes, parameters, beads (metres), the state on the device, the step."""
    g = np.random.default_rng([2401, int(seed)])
    if case["kind"] == "vessel":
        w = I.macro_case(case["n3"], MODELS[case["model"]], REACTIONS[case["reaction"]], "small", seed=int(g.integers(1 << 30)))
        shape, h, p, beads, cap = w.shape, w.h, dict(w.params), w.spheres, w.x3_cap
        cold, warm, front = -25.0, 15.0, float(g.uniform(0.35, 0.5))
    else:
        shape, cap = (case["n1"], case["n2"], case["n3"]), math.nan
        if case["model"] == "micro":
            h = 5e-8
            p = I.default_params(xi=h, xi_G=0.4 * h, zeta=2.0, theta_micro=-0.5)
            beads = packing(shape, 0.4, 6.0, 9.0, g) * h
        else:
            h = 3e-4
            p = I.default_params(xi=h, xi_G=0.4 * h, zeta=2.0, alpha=I.ALPHA_MACRO["large"],
                                 dirichlet_faces=I.FACE_ZP, theta_freeze=-5.0, theta_thaw=2.0)
            beads = packing(shape, 0.6, 10.0, 16.0, g) * h
        cold, warm, front = -5.0, 1.0, float(g.uniform(0.45, 0.55))
    if case["model"] == "micro":
        solid = surface_distance(shape, beads / h, 2.0) < 0
        phi = ball_state(shape, [n * g.uniform(0.4, 0.6) for n in shape], min(shape) / 4.0, 1.0, solid)
        theta, dt = None, 0.1 * p["alpha"] * h * h
    else:
        solid = surface_distance(shape, beads / h, 2.0) < 0
        if not math.isnan(cap):
            solid[math.floor(cap / h):] = True
        theta, phi = front_state(shape, h, p["xi"], solid, front, cold, warm)
        if case["model"] == "temp":
            phi = None
        d_ice = p["lambda"][1] / (p["rho"][1] * p["c"][1])
        dt = 1.0 / (12.0 * d_ice / (h * h) + 12.0 / (p["alpha"] * h * h))
    return shape, h, p, beads, cap, theta, phi, dt


def instances(case, seed):
    """Micro-scale instances of uneven size, each with its own packing, supercooling and surface-tension scale."""
    g = np.random.default_rng([1672, int(seed)])
    h, out = 1e-7, []
    for q in range(case["count"]):
        n = case["lo"] + 8 * round((case["hi"] - case["lo"]) * q / max(1, case["count"] - 1) / 8)
        shape = (n, n, n)
        dT, scale = float(g.choice(I.SUPERCOOLINGS[2:6])), float(g.choice(I.SIGMA_SCALES[:4]))
        p = I.default_params(xi=h, xi_G=0.4 * h, zeta=2.0, theta_micro=-dT, alpha=I.TABLE1["alpha"] / scale)
        beads = packing(shape, 0.6, 10.0, 16.0, g)
        d = surface_distance(shape, beads, 8.0)
        phi = ball_state(shape, g.uniform(0.4, 0.6, 3) * n, n / 4.0, 1.0, d < 0) * torch.sigmoid(2.0 * d - 4.0)
        # a step the tolerance always admits; in the binary32 form it is also the cap, so every instance takes
        # `steps` steps whatever the rounding noise of its error estimate
        dt = 0.03 * p["alpha"] * h * h / (1.0 + 4.0 * dT / scale)
        if case["prec"] == "f32":
            p["dt_max"] = dt
        out.append((shape, h, p, beads * h, phi, dt, (case["steps"] - 0.5) * dt, 20 * h / (p["mu"] * dT)))
    return out


def crops(case, seed):
    """Glass fields of micro-scale crops, network features and a phase field to learn."""
    g = np.random.default_rng([64, int(seed)])
    b, s = case["batch"], case["side"]
    G = torch.empty((b, s, s, s), dtype=torch.float32, device=DEV)
    feat = []
    for q in range(b):
        d = surface_distance((s, s, s), packing((s, s, s), 0.5, 10.0, 16.0, g), 6.0)
        G[q] = (0.5 * (1.0 - torch.tanh(d / 0.8))).float()
        feat.append(NN.features(float(g.uniform(0.5, 5.0)), float(g.uniform(1.0, 10.0))))
    return G, torch.tensor(feat, dtype=torch.float32, device=DEV), ((G < 0.5).float() * 0.9 + 0.05)


def layer(case, seed):
    """Activations after a ReLU and He-normal weights of one convolution layer, bfloat16."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    n, s, ci, co = case["n"], case["side"], case["cin"], case["cout"]
    x = torch.randn((n, s, s, s, ci), generator=g, device=DEV).relu_().to(torch.bfloat16)
    w = (torch.randn((27, co, ci), generator=g, device=DEV) * math.sqrt(2.0 / (27 * ci))).to(torch.bfloat16)
    return x, w, torch.randn(co, generator=g, device=DEV) * 0.1


def prediction(case, seed):
    """A predicted phase field (near 1 in the pores, noisy), the bottom-plane seed and the glass field."""
    g = np.random.default_rng([7, int(seed)])
    shape = (case["n1"], case["n2"], case["n3"])
    d = surface_distance(shape, packing(shape, 0.5, 10.0, 16.0, g), 6.0)
    G = 0.5 * (1.0 - torch.tanh(d / 0.8))
    noise = torch.rand(d.shape, generator=torch.Generator(device=DEV).manual_seed(int(seed)), device=DEV)
    prob = torch.where(d > 0.5, 0.55 + 0.45 * noise, 0.4 * noise).float()
    seed_phi = torch.zeros_like(G)
    seed_phi[0] = 1.0
    return shape, prob.reshape(-1), seed_phi.reshape(-1), G.reshape(-1).contiguous()


# ------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("grid", "vessel"):
        shape, h, p, beads, cap, theta, phi, dt = problem(case, seed)
        g = pf.Grid(shape, h, MODELS[case["model"]], REACTIONS[case["reaction"]], PRECISIONS[case["prec"]], p)
        g.set_geometry(beads, cap)
        s.update(grid=g, dt=dt, theta=None if theta is None else pinned(theta), phi=None if phi is None else pinned(phi),
                 theta_out=torch.empty(g.N, dtype=torch.float64, pin_memory=True),
                 phi_out=torch.empty(g.N, dtype=torch.float64, pin_memory=True))
        if case["tuned"]:
            g.set_state(s["theta"], s["phi"], 0.0, dt)
            g.autotune()
    elif kind == "batch":
        stream = torch.cuda.Stream()
        grids, phis, outs, inst = [], [], [], instances(case, seed)
        for shape, h, p, beads, phi, dt, t_end, window in inst:
            g = pf.Grid(shape, h, I.MODEL_MICRO, I.REACT_SIGMAP1P, PRECISIONS[case["prec"]], p, stream=stream)
            g.set_geometry(beads)
            grids.append(g)
            phis.append(pinned(phi))
            outs.append(torch.empty(g.N, dtype=torch.float64, pin_memory=True))
        rate = [1e-3 * p["mu"] * -p["theta_micro"] / (4 * p["xi"]) for _, _, p, *_ in inst]
        s.update(batch=pf.Batch(grids), grids=grids, phi=phis, out=outs, dt=[i[5] for i in inst], t_end=[i[6] for i in inst],
                 window=[i[7] for i in inst], rate=rate)
        if case["tuned"]:
            for g, phi, dt in zip(grids, phis, s["dt"]):
                g.set_state(None, phi, 0.0, dt)
            s["batch"].autotune()
    elif kind in ("train", "infer"):
        G, feat, target = crops(case, seed)
        s.update(net=NN.UNet(seed=int(seed) % 1000), G=G.reshape(-1), feat=feat, target=target.reshape(-1))
    elif kind == "conv":
        x, w, b = layer(case, seed)
        y = torch.empty(x.shape[:4] + (case["cout"],), dtype=torch.bfloat16, device=DEV)
        s.update(x=x, w=w, b=b, y=y, lib=NN._lib())
    else:
        shape, prob, phi, G = prediction(case, seed)
        s.update(shape=shape, prob=prob, phi=phi, G=G)
    torch.cuda.synchronize()
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("grid", "vessel"):
        g = state["grid"]
        g.set_state(state["theta"], state["phi"], 0.0, state["dt"])
        if case["adaptive"]:
            st = g.run_to(1e30, 1e-6, case["steps"])
        else:
            st = g.run_fixed(case["steps"], state["dt"])
        if case["model"] == "micro":  # the host program knows its constant temperature
            _get_phi(g, state["phi_out"])
            out = [state["phi_out"]]
        else:
            g.get_state(state["theta_out"], state["phi_out"])
            out = [state["theta_out"], state["phi_out"]]
        return out + [st["t"], st["n_accepted"], st["n_rejected"]]
    if kind == "batch":
        for g, phi, dt in zip(state["grids"], state["phi"], state["dt"]):
            g.set_state(None, phi, 0.0, dt)
        if case["prec"] == "f32":
            res = state["batch"].run_to(state["t_end"], 1e-6, 100000)
        else:  # adaptive to the equilibrium test or the attempt cap
            res = state["batch"].run_to([1e30] * len(state["dt"]), 1e-6, case["steps"], state["window"], 1e-3, state["rate"])
        for g, out in zip(state["grids"], state["out"]):
            _get_phi(g, out)
        return state["out"] + [[r["t"] for r in res], [r["n_accepted"] + r["n_rejected"] for r in res]]
    if kind == "train":
        net = state["net"]
        prob = net.forward(state["G"], state["feat"], state["target"])
        net.backward()
        net.adam_step(lr=2e-9)  # the end of the cosine decay
        grads = [net.get_grads(name) for name in net.names]
        return [prob, net.loss_value(), [w for w, _ in grads], [b for _, b in grads]]
    if kind == "infer":
        return state["net"].forward(state["G"], state["feat"])
    if kind == "conv":
        x, w, b, y = state["x"], state["w"], state["b"], state["y"]
        n, s, ci, co = case["n"], case["side"], case["cin"], case["cout"]
        NN._ck(state["lib"].pfnn_conv3d(NN._p(x), ci, 0, NN._p(w), ci, co, NN._p(b), 1, 0, NN._p(y), None, co, 0, 0, n, s,
                                        s, s, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)), "conv3d")
        return y
    return NN.seed_connect(state["prob"], state["phi"], state["G"], state["shape"], 2.0)[0]


def _get_phi(g, out):
    """pf_get_state without the (constant) temperature of the micro model."""
    pf._check(pf.load_library().pf_get_state(g.handle, None, out.data_ptr(), None, None), g.handle)


# ------------------------------------------------------------------ work
# flops of one right-hand side and the five stage combinations per cell, as the method writes them (full model with
# the sigma-limited reaction): blends 18, fluxes 24, Allen-Cahn 16, coupling 6; combinations 4 + 6 + 8 + 12 + 24
FLOPS = {"full": 5 * 64 + 54, "temp": 5 * 66 + 27, "micro": 5 * 16 + 27}
# bytes per cell and attempt with every field of a stage read and written once (state, slopes and stage inputs, glass)
BYTES = {("full", "f64"): 424, ("full", "f32"): 252, ("temp", "f64"): 232, ("temp", "f32"): 136, ("micro", "f64"): 232,
         ("micro", "f32"): 136}

# the network's convolutions: (level, cin, cout)
CONVS = [(0, 16, 16), (0, 16, 16), (1, 16, 32), (1, 32, 32), (2, 32, 64), (2, 64, 64), (3, 64, 128), (3, 128, 128),
         (2, 128, 64), (2, 128, 64), (2, 64, 64), (1, 64, 32), (1, 64, 32), (1, 32, 32), (0, 32, 16), (0, 32, 16),
         (0, 16, 16)]


def work(case):
    kind = case["kind"]
    if kind in ("grid", "vessel", "batch"):
        if kind == "batch":
            model = "micro"
            sizes = [case["lo"] + 8 * round((case["hi"] - case["lo"]) * q / max(1, case["count"] - 1) / 8)
                     for q in range(case["count"])]
            n = float(sum(s ** 3 for s in sizes))
        else:
            model = case["model"]
            n = float(case["n3"] ** 3 / 4 if kind == "vessel" else case["n1"] * case["n2"] * case["n3"])
        return {"bytes": n * case["steps"] * BYTES[model, case["prec"]], "flops": n * case["steps"] * FLOPS[model]}
    if kind in ("train", "infer"):
        v = float(case["batch"] * case["side"] ** 3)
        fl = sum(2 * 27 * ci * co * v / 8 ** lev for lev, ci, co in CONVS)
        io = sum(2 * (ci + co) * v / 8 ** lev for lev, ci, co in CONVS)
        if kind == "infer":
            return {"bytes": io + 8 * v, "flops": fl}
        first = 2 * 27 * 16 * 16 * v  # no gradient for the network's input
        return {"bytes": 3 * io + 12 * v, "flops": 3 * fl - first}
    if kind == "conv":
        v = float(case["n"] * case["side"] ** 3)
        return {"bytes": 2 * v * (case["cin"] + case["cout"]) + 54 * case["cin"] * case["cout"],
                "flops": 54 * v * case["cin"] * case["cout"]}
    v = float(case["n1"] * case["n2"] * case["n3"])
    return {"bytes": v * (4 + 8 + 8 + 8), "flops": 0}


# ------------------------------------------------------------------ binary64 reference in plain torch
def _pad(a):
    return torch.nn.functional.pad(a[None, None], (1, 1, 1, 1, 1, 1), mode="replicate")[0, 0]


def _rhs(m, theta, phi, t):
    """Right-hand side of Secs. 2.2-2.4 (eqs. heat-equation, Allen-Cahn-equation, combined-heat-xfer-phase-transition)
    by finite volumes, arithmetic face means."""
    p, h, G = m["p"], m["h"], m["G"]
    iw = torch.clamp(1.0 - p["zeta"] * G, min=0.0)
    if m["model"] == "temp":
        tg = torch.tanh(p["gamma"] * theta)
        phi = 0.5 * iw * (1.0 - tg)

    def blend(w):
        return w[0] + G * (w[2] - w[0]) + (1.0 - G) * phi * (w[1] - w[0])

    def shifted(a):
        q = _pad(a)
        return (q[1:-1, 1:-1, :-2], q[1:-1, 1:-1, 2:], q[1:-1, :-2, 1:-1], q[1:-1, 2:, 1:-1], q[:-2, 1:-1, 1:-1],
                q[2:, 1:-1, 1:-1])

    div = 0.0
    if m["model"] != "micro":
        lam = blend(p["lambda"])
        for l, th in zip(shifted(lam), shifted(theta)):
            div = div + 0.5 * (lam + l) * (th - theta)
        if p["dirichlet_faces"] & I.FACE_ZP:
            wall = p["theta_freeze"] if t < p["t_freeze"] else p["theta_thaw"]
            div[-1] += 2.0 * lam[-1] * (wall - theta[-1])
        div = div / (h * h)
        rho, c = blend(p["rho"]), blend(p["c"])
        if m["model"] == "temp":
            dp = -0.5 * iw * p["gamma"] * (1.0 - tg * tg)
            return div / (rho * (c - p["latent"] * dp)), None
    th = p["theta_micro"] if m["model"] == "micro" else theta
    nb = shifted(phi)
    lap = (sum(nb) - 6.0 * phi) / (h * h)
    if m["reaction"] == "gradp":
        gn = torch.sqrt((nb[1] - nb[0]) ** 2 + (nb[3] - nb[2]) ** 2 + (nb[5] - nb[4]) ** 2) / (2.0 * h)
        f = 2.0 * phi * (1.0 - phi) * (phi - 0.5) - p["xi"] ** 2 * p["mu"] * p["alpha"] * gn * th
    else:
        def lim(w):
            s = torch.clamp((w - p["eps0"]) / (p["eps1"] - p["eps0"]), 0.0, 1.0)
            return s * s * (3.0 - 2.0 * s)

        S = lim(phi) * lim(1.0 - phi)
        f = 2.0 * phi * (1.0 - phi) * (phi - 0.5 - 0.5 * p["xi"] * p["b"] * p["mu"] * p["alpha"] * S * th)
    dphi = iw / (p["alpha"] * p["xi"] ** 2) * (p["xi"] ** 2 * lap + f)
    if m["model"] == "micro":
        return None, dphi
    return (div + p["latent"] * rho * dphi) / (rho * c), dphi


def _integrate(m, theta, phi, dt, steps, tol=None, t_end=math.inf, dt_max=math.inf):
    """Runge-Kutta-Merson with the library's documented step control (fixed steps when tol is None)."""
    y = [theta, phi]
    t, acc, rej, step = 0.0, 0, 0, dt

    def F(u):
        return _rhs(m, u[0], u[1], t)

    def mix(a, *terms):
        return [None if q is None else q + a * sum(c * k[j] for c, k in terms) for j, q in enumerate(y)]

    while acc + rej < steps and t < t_end:
        land = t + step >= t_end
        d = t_end - t if land else step
        k1 = F(y)
        k2 = F(mix(d, (1 / 3, k1)))
        k3 = F(mix(d, (1 / 6, k1), (1 / 6, k2)))
        del k2
        k4 = F(mix(d, (1 / 8, k1), (3 / 8, k3)))
        k5 = F(mix(d, (1 / 2, k1), (-3 / 2, k3), (2.0, k4)))
        new = mix(d, (1 / 6, k1), (4 / 6, k4), (1 / 6, k5))
        if tol is None:
            y, t, acc = new, t + d, acc + 1
            continue
        e = max(float((d / 30 * (2 * a - 9 * b + 8 * c - k)).abs().max()) for a, b, c, k in zip(k1, k3, k4, k5)
                if a is not None)
        if e <= tol:
            y, t, acc = new, (t_end if land else t + d), acc + 1
        else:
            rej += 1
        step = min(dt_max, d * (5.0 if e == 0 else min(5.0, 0.8 * (tol / e) ** 0.2)))
    return y, t, acc, rej


class _Bf16Out(torch.autograd.Function):
    """Storage in bfloat16: the value is rounded, the gradient passes."""

    @staticmethod
    def forward(ctx, x):
        return x.to(torch.bfloat16).to(x.dtype)

    @staticmethod
    def backward(ctx, g):
        return g


class _Bf16Grad(torch.autograd.Function):
    """The gradient that enters a convolution's backward products is stored in bfloat16."""

    @staticmethod
    def forward(ctx, x):
        return x.clone()

    @staticmethod
    def backward(ctx, g):
        return g.to(torch.bfloat16).to(g.dtype)


def _conv(x, w):
    """3x3x3 convolution, zero padding, channels last; w [27][cout][cin]."""
    n, d, h, wd, _ = x.shape
    q = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    out = 0.0
    for t in range(27):
        a, b, c = t // 9, t // 3 % 3, t % 3
        out = out + q[:, a:a + d, b:b + h, c:c + wd] @ w[t].T
    return out


def _network(case, seed, grads):
    G, feat, target = crops(case, seed)
    net = NN.UNet(seed=int(seed) % 1000)  # only for its initial weights
    P = {k: [torch.from_numpy(v).to(DEV).double().requires_grad_(grads) for v in net.get_params(k)] for k in net.names}
    net.close()
    b, s = case["batch"], case["side"]
    x = torch.zeros((b, s, s, s, 16), dtype=torch.float64, device=DEV)
    x[..., 0] = G.to(torch.bfloat16).double()
    x[..., 1:3] = feat.to(torch.bfloat16).double()[:, None, None, None]

    def block(x, name):
        w, bias = P[name]
        return _Bf16Out.apply(torch.relu(_Bf16Grad.apply(_conv(x, _Bf16Out.apply(w))) + bias))

    def pool(x):
        n, d, h, w, c = x.shape
        return _Bf16Out.apply(x.reshape(n, d // 2, 2, h // 2, 2, w // 2, 2, c).mean(dim=(2, 4, 6)))

    def up(x):
        return x.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)

    with torch.set_grad_enabled(grads):
        c1 = block(block(x, "e1a"), "e1b")
        c2 = block(block(pool(c1), "e2a"), "e2b")
        c3 = block(block(pool(c2), "e3a"), "e3b")
        q = block(block(pool(c3), "e4a"), "e4b")
        q = block(block(torch.cat([c3, block(up(q), "u3")], -1), "d3a"), "d3b")
        q = block(block(torch.cat([c2, block(up(q), "u2")], -1), "d2a"), "d2b")
        q = block(block(torch.cat([c1, block(up(q), "u1")], -1), "d1a"), "d1b")
        w, bias = P["head"]
        z = (q @ w + bias).reshape(-1)
    prob = torch.sigmoid(z.detach())
    if not grads:
        return prob
    loss = torch.nn.functional.binary_cross_entropy_with_logits(z, target.double().reshape(-1))
    loss.backward()
    return [prob, float(loss), [P[k][0].grad for k in P], [P[k][1].grad for k in P]]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("grid", "vessel"):
        shape, h, p, beads, cap, theta, phi, dt = problem(case, seed)
        m = dict(p=p, h=h, G=glass(shape, h, beads, p["xi_G"], cap), model=case["model"], reaction=case["reaction"])
        y, t, acc, rej = _integrate(m, theta, phi, dt, case["steps"], 1e-6 if case["adaptive"] else None)
        if case["model"] == "temp":
            iw = torch.clamp(1.0 - p["zeta"] * m["G"], min=0.0)
            y[1] = 0.5 * iw * (1.0 - torch.tanh(p["gamma"] * y[0]))
        return [v.reshape(-1) for v in y if v is not None] + [t, acc, rej]
    if kind == "batch":
        out, ts, n = [], [], []
        for shape, h, p, beads, phi, dt, t_end, window in instances(case, seed):
            m = dict(p=p, h=h, G=glass(shape, h, beads, p["xi_G"], math.nan), model="micro", reaction="sigmap1p")
            # (no instance meets the equilibrium test within these attempts)
            y, t, acc, rej = _integrate(m, None, phi, dt, 100000 if case["prec"] == "f32" else case["steps"], 1e-6,
                                        t_end if case["prec"] == "f32" else math.inf, p["dt_max"])
            out.append(y[1].reshape(-1))
            ts.append(t)
            n.append(acc + rej)
        return out + [ts, n]
    if kind in ("train", "infer"):
        return _network(case, seed, kind == "train")
    if kind == "conv":
        x, w, b = layer(case, seed)
        return torch.relu(_conv(x.double(), w.double()) + b.double())
    # the seed constraint: the flood fill's fixed point, then the halo
    shape, prob, phi, G = prediction(case, seed)
    s3 = (case["n3"], case["n2"], case["n1"])
    water = (1.0 - 2.0 * G > 0).reshape(s3)
    mask = (prob > 0.5).reshape(s3) & water
    reached = (phi > 0.5).reshape(s3)

    def grow(a):
        o = a.clone()
        o[1:] |= a[:-1]
        o[:-1] |= a[1:]
        o[:, 1:] |= a[:, :-1]
        o[:, :-1] |= a[:, 1:]
        o[:, :, 1:] |= a[:, :, :-1]
        o[:, :, :-1] |= a[:, :, 1:]
        return o

    while True:
        nxt = reached
        for _ in range(32):
            nxt = (grow(nxt) & mask) | nxt
        if bool((nxt == reached).all()):
            break
        reached = nxt
    for _ in range(3):
        reached = grow(reached)
    p = prob.double().clamp(0, 1)
    return torch.where((water & reached).reshape(-1), torch.maximum(p, phi), phi)
