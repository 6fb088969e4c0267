"""Workloads that time the library through its public entry points.

Most cases are whole runs as a user's program makes them: initial fields in
device memory go in (the first encode), some time steps follow, and the
decoded state, the per-field FP64 sums and the compressed size come out.  The
others are the batch, the lossless stage of a checkpoint, and the two parts
of the learned threshold that run off the step path (labels, training).
"""
import math

import numpy as np
import torch

from paper_2302_09883_gb300 import Batch, Sim, Sim3, learned

DEV = "cuda"
FIELDS = {"d2q9": 9, "euler2d": 4, "transport": 1, "swe": 3, "d3q19": 19}


def _run(name, scheme, nx, ny, P, L, eps, steps, **kw):
    c = dict(name=name, kind="run", scheme=scheme, wavelet="bl53", nx=nx, ny=ny, nz=1, P=P, L=L, eps=eps, steps=steps,
             prec="f32", store="bf16", rule="const", init="shear", periodic=True, tau=0.6, cfl=0.4, arena=0.0,
             hilo=False, mode="uniform")
    c.update(kw)
    return c


def listed():
    return [
        # the smallest run: 16 Haar patches in FP64, a bump that spreads; launch and latency bound
        _run("haar_128_f64", "d2q9", 128, 128, 32, 3, 1e-4, 100, wavelet="haar", prec="f64", store="f64", init="bump",
             tau=0.8, arena=1.5),
        # the ordinary LBM run: noisy shear wave, BF16 details, error within 1e-3
        _run("d2q9_2048_bf16", "d2q9", 2048, 2048, 64, 4, 1e-3, 40),
        # an odd, non-square grid with FP32 details at a small threshold: most words hold survivors
        _run("d2q9_1088x704_f32", "d2q9", 1088, 704, 64, 4, 3e-7, 40, store="f32", rule="accum"),
        # compressible flow with shocks, outflow borders, int8 details, dt from the CFL condition
        _run("euler_4096_i8", "euler2d", 4096, 4096, 64, 4, 1e-4, 16, store="i8", init="quadrants", periodic=False),
        # linear transport on a ragged outflow grid, the capped rule
        _run("transport_2112x1600", "transport", 2112, 1600, 64, 4, 0.01, 64, store="f32", rule="capped",
             init="transport", periodic=False, cfl=0.45),
        # the shallow-water cost study: 129^2 nodes, few patches, many cheap steps
        _run("swe_128", "swe", 128, 128, 32, 4, 5e-4, 200, store="f32", rule="capped", init="square", periodic=False,
             cfl=-128 * 10.0 / 38245),
        # many independent grids of uneven sizes stepped together, FP32 details
        dict(name="batch_16", kind="batch", n256=6, n512=6, n1024=3, n2048=1, eps=1e-6, store="f32", tau=0.6, steps=60),
        # 3-D vortex, the ordinary cubic patches with BF16 details
        _run("d3q19_256_bf16", "d3q19", 256, 256, 32, 3, 1e-7, 6, nz=256, init="vortex", tau=0.55),
        # 3-D on a small ragged box: 16-cell patches, FP32 details
        _run("d3q19_176x80x112_f32", "d3q19", 176, 80, 16, 3, 1e-6, 12, nz=112, store="f32", init="vortex", tau=0.55),
        # features and labels of one dense snapshot (training data of the per-patch threshold)
        dict(name="labels_512", kind="labels", nx=512, ny=512, nz=1, P=64, L=4, delta=1e-5),
        # training that network on the gathered samples
        dict(name="fit_2048", kind="fit", n=2048, nin=24, epochs=10, batch=128),
        # checkpoint: entropy-coding the records of a state some way into a run
        dict(name="checkpoint_2048", kind="code", nx=2048, ny=2048, P=64, L=4, eps=1e-7, store="bf16", tau=0.6,
             steps=200),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _multiple(rng, P, lo, hi):
    """A multiple of P, log-uniform in [lo, hi] cells."""
    return max(1, round(_log(rng, lo, hi) / P)) * P


def draw(rng):
    kind = rng.choice(["d2q9", "d2q9", "d2q9", "euler2d", "euler2d", "transport", "swe", "d3q19", "d3q19", "batch",
                       "labels", "labels3", "fit", "code"])
    if kind == "d2q9":
        wavelet, prec, store, P, L = rng.choice([("bl53", "f32", "bf16", 64, 4), ("bl53", "f32", "bf16", 32, 3),
                                                 ("bl53", "f32", "f32", 64, 4), ("bl53", "f32", "f32", 32, 3),
                                                 ("bl53", "f32", "i8", 64, 4), ("bl53", "f64", "f64", 32, 3),
                                                 ("haar", "f64", "f64", 32, 3)])
        top = 1024 if prec == "f64" else 2048
        # hi + lo coarse storage and per-patch thresholds (given, or from a network) now and then
        mode = rng.choice(["uniform", "uniform", "uniform", "patch_eps", "network"])
        c = _run("", "d2q9", _multiple(rng, P, 96, top), _multiple(rng, P, 96, top), P, L, _log(rng, 1e-7, 1e-3),
                 rng.randint(8, 60), wavelet=wavelet, prec=prec, store=store,
                 rule=rng.choice(["const", "accum", "capped"]), init=rng.choice(["shear", "bump"]),
                 tau=round(rng.uniform(0.55, 0.9), 3), arena=1.5, mode=mode,
                 hilo=mode == "uniform" and prec == "f32" and rng.random() < 0.2)
    elif kind == "euler2d":
        prec, store, P, L = rng.choice([("f32", "i8", 64, 4), ("f32", "bf16", 64, 4), ("f64", "f64", 32, 3)])
        top = 1024 if prec == "f64" else 4096
        c = _run("", "euler2d", _multiple(rng, P, 128, top), _multiple(rng, P, 128, top), P, L, _log(rng, 1e-5, 1e-3),
                 rng.randint(4, 16), prec=prec, store=store, init="quadrants", periodic=rng.random() < 0.3,
                 cfl=rng.choice([0.4, 0.4, -0.1]), arena=1.5)
    elif kind == "transport":
        wavelet, prec, P, L = rng.choice([("bl53", "f32", 64, 1), ("bl53", "f32", 64, 2), ("bl53", "f32", 64, 3),
                                          ("bl53", "f32", 64, 4), ("bl53", "f32", 64, 5), ("cdf97", "f32", 64, 4),
                                          ("bl53", "f64", 32, 3)])
        c = _run("", "transport", _multiple(rng, P, 128, 4096), _multiple(rng, P, 128, 4096), P, L,
                 rng.uniform(0.002, 0.05), rng.randint(16, 64), wavelet=wavelet, prec=prec,
                 store="f64" if prec == "f64" else "f32", rule=rng.choice(["const", "accum", "capped"]),
                 init="transport", periodic=rng.random() < 0.3, cfl=0.45, arena=1.5)
    elif kind == "swe":
        prec, P, L = rng.choice([("f32", 64, 4), ("f32", 32, 4), ("f64", 32, 3)])
        c = _run("", "swe", _multiple(rng, P, 128, 1024), _multiple(rng, P, 128, 1024), P, L, _log(rng, 1e-4, 1e-3),
                 rng.randint(10, 40), prec=prec, store="f64" if prec == "f64" else "f32", rule="capped", init="square",
                 periodic=rng.random() < 0.3, cfl=rng.choice([0.4, -0.03]), arena=1.5)
    elif kind == "d3q19":
        P = rng.choice([32, 32, 16])
        lo, hi = (32, 288) if P == 32 else (32, 160)
        c = _run("", "d3q19", _multiple(rng, P, lo, hi), _multiple(rng, P, lo, hi), P, 3, _log(rng, 1e-7, 1e-5),
                 rng.randint(3, 6), nz=_multiple(rng, P, lo, hi), store=rng.choice(["bf16", "bf16", "f32"]),
                 init="vortex", tau=round(rng.uniform(0.52, 0.8), 3), arena=1.5)
        if rng.random() < 0.15:
            c["hilo"] = True
    elif kind == "batch":
        c = dict(kind="batch", n256=rng.randint(1, 8), n512=rng.randint(0, 6), n1024=rng.randint(0, 3), n2048=1,
                 eps=_log(rng, 1e-7, 1e-4), store=rng.choice(["f32", "bf16"]), tau=round(rng.uniform(0.55, 0.9), 3),
                 steps=rng.randint(6, 60))
    elif kind == "labels":
        c = dict(kind="labels", nx=_multiple(rng, 64, 64, 640), ny=_multiple(rng, 64, 64, 512), nz=1, P=64, L=4,
                 delta=_log(rng, 1e-6, 1e-4))
    elif kind == "labels3":
        c = dict(kind="labels", nx=32 * rng.randint(1, 4), ny=32 * rng.randint(1, 4), nz=32 * rng.randint(1, 4),
                 P=rng.choice([32, 32, 16]), L=3, delta=_log(rng, 3e-7, 3e-5))
    elif kind == "fit":
        c = dict(kind="fit", n=rng.randint(192, 2048), nin=rng.choice([18, 24, 42]), epochs=rng.randint(2, 10),
                 batch=rng.choice([32, 64, 100, 128]))
    else:
        c = dict(kind="code", nx=_multiple(rng, 64, 128, 2048), ny=_multiple(rng, 64, 128, 2048), P=64, L=4,
                 eps=_log(rng, 1e-7, 1e-4), store=rng.choice(["bf16", "f32"]), tau=0.6, steps=rng.randint(50, 250))
    c.pop("name", None)
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(1 + seed)


def _rand(seed, k):
    return np.random.default_rng([seed, 77]).uniform(0.0, 1.0, k)


def _axes(c):
    """Node counts: an outflow axis carries its last node too (nodal wavelets)."""
    extra = 0 if c["periodic"] or c["wavelet"] == "haar" else 1
    return c["nx"] + extra, c["ny"] + extra


def _fields(c, seed):
    """Initial macroscopic fields (float64 device tensors) from the seed."""
    r = _rand(seed, 8)
    if c["init"] == "vortex":  # Taylor-Green vortex, seeded strength and phase, a little noise in the velocity
        k = [2.0 * math.pi * torch.arange(n, dtype=torch.float64, device=DEV) / n + 2.0 * math.pi * p
             for n, p in zip((c["nx"], c["ny"], c["nz"]), r)]
        x, y, z = k[0][None, None, :], k[1][None, :, None], k[2][:, None, None]
        u0 = 0.02 + 0.04 * r[3]
        ux = u0 * torch.sin(x) * torch.cos(y) * torch.cos(z)
        uy = -u0 * torch.cos(x) * torch.sin(y) * torch.cos(z)
        g = _gen(seed)
        noise = lambda: 1e-6 * torch.randn(ux.shape, generator=g, device=DEV, dtype=torch.float64)
        rho = 1.0 + 3.0 * u0 * u0 / 16.0 * (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0)
        return [rho.contiguous(), ux + noise(), uy + noise(), noise()]
    gx, gy = _axes(c)
    i = torch.arange(gx, dtype=torch.float64, device=DEV)[None, :]
    j = torch.arange(gy, dtype=torch.float64, device=DEV)[:, None]
    if c["init"] == "bump":  # density bump at rest
        sig = min(4.0 + 28.0 * r[0], min(gx, gy) / 12.0)
        rho = 1.0 + (0.01 + 0.09 * r[1]) * torch.exp(-((i - gx * r[2]) ** 2 + (j - gy * r[3]) ** 2) / (2 * sig * sig))
        return [rho, torch.zeros_like(rho), torch.zeros_like(rho)]
    if c["init"] == "shear":  # shear wave with noise in u_x
        n = torch.randn((gy, gx), generator=_gen(seed), device=DEV, dtype=torch.float64)
        ux = (0.03 + 0.02 * r[0]) * torch.sin(2 * math.pi * (j / gy + r[1])) + 1e-4 * n
        return [torch.ones_like(ux), ux, torch.zeros_like(ux)]
    x, y = i / c["nx"], j / c["ny"]
    if c["init"] == "quadrants":  # four-quadrant Riemann data plus smooth waves: shocks and a structured background
        e, n = (x >= 0.4 + 0.2 * r[0]), (y >= 0.4 + 0.2 * r[1])
        pick = lambda sw, se, nw, ne: torch.where(n, torch.where(e, ne, nw), torch.where(e, se, sw)).double()
        q = lambda *v: pick(*[torch.tensor(t, dtype=torch.float64, device=DEV) for t in v])
        wave = 1.0 + 0.02 * torch.sin(2 * math.pi * (6 * x + r[2])) * torch.sin(2 * math.pi * (5 * y + r[3]))
        return [q(0.138, 0.5323, 0.5323, 1.5) * wave, q(1.206, 0.0, 1.206, 0.0), q(1.206, 1.206, 0.0, 0.0),
                q(0.029, 0.3, 0.3, 1.5) * wave]
    if c["init"] == "transport":  # Gaussian on [-1, 1]^2
        w = 1.0 + torch.exp(-(20.0 + 20.0 * r[0]) * ((2 * x - 1 - 0.3 * r[1]) ** 2 + (2 * y - 1 + 0.3 * r[2]) ** 2))
        return [w.contiguous()]
    half, cx, cy = 0.15 + 0.1 * r[0], 0.45 + 0.1 * r[1], 0.45 + 0.1 * r[2]  # raised square of water at rest
    h = torch.where(((x - cx).abs() <= half) & ((y - cy).abs() <= half), 1.5 + r[3], 1.0).double()
    return [h.contiguous(), torch.zeros_like(h), torch.zeros_like(h)]


def _velocity(seed):
    r = _rand(seed, 8)
    return 0.6 + 0.3 * float(r[4]), 0.6 + 0.3 * float(r[5])


def _batch_list(c):
    return [n for n, key in ((2048, "n2048"), (1024, "n1024"), (512, "n512"), (256, "n256")) for _ in range(c[key])]


def _snapshot(c, seed):
    """A dense FP32 LBM state: equilibrium of smooth waves plus noise whose
    amplitude changes from patch to patch."""
    g, P, nx, ny, nz = _gen(seed), c["P"], c["nx"], c["ny"], c["nz"]
    three = nz > 1
    shape = (nz, ny, nx) if three else (ny, nx)
    k = [2 * math.pi * torch.arange(n, dtype=torch.float64, device=DEV) / n for n in shape]
    grids = torch.meshgrid(*k, indexing="ij")
    amp = 10.0 ** (-7.0 + 5.0 * torch.rand([n // P for n in shape], generator=g, device=DEV, dtype=torch.float64))
    for d in range(len(shape)):
        amp = amp.repeat_interleave(P, d)
    noise = lambda: amp * torch.randn(shape, generator=g, device=DEV, dtype=torch.float64)
    p = _rand(seed, 8) * 2 * math.pi
    u = [0.04 * torch.sin(grids[-2] + p[0]) + noise(), 0.02 * torch.sin(grids[-1] + p[1]) + noise()]
    rho = 1.0 + 0.01 * torch.sin(grids[-1] + p[2]) * torch.sin(grids[-2] + p[3])
    u += [0.01 * torch.sin(grids[-1] + p[4]) + noise()] if three else []
    return torch.stack(_equilibrium(rho, u, *(_D3 if three else _D2))).float().contiguous()


def _samples(c, seed):
    """Features (log10 energies and maxima) and labels (log10 eps) of n patches."""
    g = _gen(seed)
    base = torch.randn((c["n"], 3), generator=g, device=DEV)
    mix = torch.randn((3, c["nin"]), generator=g, device=DEV)
    X = -8.0 + 2.0 * base @ mix + 0.3 * torch.randn((c["n"], c["nin"]), generator=g, device=DEV)
    t = -4.5 + torch.tanh(base[:, 0]) + 0.5 * base[:, 1] * base[:, 2].sigmoid()
    return X.contiguous(), t.contiguous()


# --------------------------------------------------------------- the calls
def _sim(c, seed):
    if c["scheme"] == "d3q19":
        return Sim3(c["nx"], c["ny"], c["nz"], c["P"], c["L"], c["eps"], store=c["store"], rule=c["rule"], tau=c["tau"],
                    arena_factor=c["arena"], coarse_hilo=c["hilo"])
    per = c["periodic"]
    return Sim(c["scheme"], c["wavelet"], c["nx"], c["ny"], c["P"], c["L"], c["eps"], prec=c["prec"], store=c["store"],
               rule=c["rule"], periodic=(per, per), tau=c["tau"], cfl=c["cfl"], arena_factor=c["arena"],
               velocity=_velocity(seed), length=2.0 if c["scheme"] == "transport" else 1.0, coarse_hilo=c["hilo"])


def _out(sim, prec):
    shape = (sim.F,) + tuple(reversed(sim.G))
    return torch.empty(shape, dtype=torch.float64 if prec == "f64" else torch.float32, device=DEV)


def prepare(case, seed):
    c, s = case, {"case": case, "seed": seed}
    if c["kind"] == "run":
        s["fields"] = _fields(c, seed)
        s["sim"] = _sim(c, seed)
        s["out"] = _out(s["sim"], c["prec"])
        if c["mode"] == "patch_eps":
            r = np.random.default_rng([seed, 5])
            learned.set_patch_eps(s["sim"], c["eps"] * 10.0 ** r.uniform(-1.0, 1.0, s["sim"].npatch))
        elif c["mode"] == "network" and c["wavelet"] == "bl53":
            s["net"] = learned.Mlp(6 * c["L"], seed=seed)
            learned.use_mlp(s["sim"], s["net"], 0.1 * c["eps"], 10.0 * c["eps"])
    elif c["kind"] == "batch":
        s["sims"], s["fields"], s["out"] = [], [], []
        for k, n in enumerate(_batch_list(c)):
            P, L = (64, 4) if n >= 1024 else (32, 3)
            one = _run("", "d2q9", n, n, P, L, c["eps"], 0, store=c["store"], tau=c["tau"], init="bump", arena=1.5)
            s["fields"].append(_fields(one, 1000 * seed + k))
            s["sims"].append(_sim(one, seed))
            s["out"].append(_out(s["sims"][-1], "f32"))
    elif c["kind"] == "labels":
        s["dense"] = _snapshot(c, seed)
    elif c["kind"] == "fit":
        s["X"], s["t"] = _samples(c, seed)
    else:
        one = _run("", "d2q9", c["nx"], c["ny"], c["P"], c["L"], c["eps"], 0, store=c["store"], tau=c["tau"])
        s["sim"] = _sim(one, seed)
        s["sim"].init_macro(_fields(one, seed))
        s["sim"].step(c["steps"])
        s["sim"].sync()
        s["file"], s["used"] = np.zeros(9 * 4 * c["nx"] * c["ny"] // 2, np.uint8), 0  # where the checkpoint goes
    return s


def _export(sim, out):
    return sim.export_field(-1, out=out, dtype=np.float64 if out.dtype == torch.float64 else np.float32)


def run(state):
    c = state["case"]
    if c["kind"] == "run":
        sim = state["sim"]
        if "net" in state:  # a run of its own starts from the uniform eps
            learned.use_mlp(sim, state["net"], 0.1 * c["eps"], 10.0 * c["eps"])
        sim.init_macro(state["fields"])
        sim.step(c["steps"])
        st = sim.stats()
        return {"state": _export(sim, state["out"]), "field_sum": st["field_sum"], "time": st["time"],
                "bytes": sim.compressed_bytes()}
    if c["kind"] == "batch":
        sims = state["sims"]
        for sim, f in zip(sims, state["fields"]):
            sim.init_macro(f)
        b = Batch(sims)
        b.step(c["steps"])
        b.sync()
        b.close()
        return {"states": [_export(sim, out) for sim, out in zip(sims, state["out"])],
                "bytes": [sim.compressed_bytes() for sim in sims]}
    if c["kind"] == "labels":
        fn = learned.features_labels3 if c["nz"] > 1 else learned.features_labels
        feat, label = fn(state["dense"], c["P"], c["L"], c["delta"])
        return {"features": feat, "labels": label}
    if c["kind"] == "fit":
        net, hist = learned.fit(state["X"], state["t"], epochs=c["epochs"], batch=c["batch"], seed=state["seed"])
        return {"weights": net.weights(), "loss": hist}
    coded, file = np.frombuffer(state["sim"].entropy_code(), dtype=np.uint8), state["file"]
    file[:len(coded)] = coded
    file[len(coded):state["used"]] = 0
    state["used"] = len(coded)
    return {"file": file, "bytes": len(coded)}


def _lift_flops(L):
    return sum(3.5 / 2 ** k for k in range(L))  # one axis, one direction, per node: 3 per detail, 4 per even node


_SCHEME_FLOPS = {"d2q9": 135, "d3q19": 330, "euler2d": 180, "transport": 14, "swe": 600}


def _run_work(c):
    dims = 3 if c["scheme"] == "d3q19" else 2
    F, nodes = FIELDS[c["scheme"]], c["nx"] * c["ny"] * c["nz"]
    tb = 8 if c["prec"] == "f64" else 4
    nin = {"d2q9": 3, "d3q19": 4, "euler2d": 4, "transport": 1, "swe": 3}[c["scheme"]]
    coarse = nodes // c["P"] ** dims * F * ((c["P"] >> c["L"]) + (c["wavelet"] != "haar")) ** dims * tb
    lift = F * dims * _lift_flops(c["L"])
    return {"bytes": 8 * nin * nodes + tb * F * nodes + 2 * c["steps"] * coarse,
            "flops": nodes * (2 * lift + c["steps"] * (2 * lift + _SCHEME_FLOPS[c["scheme"]]))}


def work(case):
    c = case
    if c["kind"] == "run":
        return _run_work(c)
    if c["kind"] == "batch":
        each = [_run_work(_run("", "d2q9", n, n, *((64, 4) if n >= 1024 else (32, 3)), c["eps"], c["steps"]))
                for n in _batch_list(c)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    if c["kind"] == "labels":
        F, dims = (19, 3) if c["nz"] > 1 else (9, 2)
        nodes = c["nx"] * c["ny"] * c["nz"]
        # the forward transform, and one inverse per probed eps: a search of the 41-value grid and four bisections
        return {"bytes": 4 * F * nodes, "flops": F * nodes * dims * _lift_flops(c["L"]) * (1 + 6 + 4)}
    if c["kind"] == "fit":
        par = 64 * c["nin"] + 64 + 64 * 64 + 64 + 64 + 1
        seen = c["epochs"] * (c["n"] // c["batch"]) * c["batch"]
        return {"bytes": 4 * c["n"] * (c["nin"] + 1) + 4 * par, "flops": 6 * par * seen}
    npatch = c["nx"] * c["ny"] // c["P"] ** 2
    return {"bytes": 2 * npatch * 9 * ((c["P"] >> c["L"]) + 1) ** 2 * 4, "flops": 0}


# ------------------------------------------------- the same in 64 bits
_CX = [0, 1, 0, -1, 0, 1, -1, -1, 1]
_CY = [0, 0, 1, 0, -1, 1, 1, -1, -1]
_D2 = (list(zip(_CX, _CY)), [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
_D3 = ([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
        (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
        (0, -1, 1)], [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


def _equilibrium(rho, u, vel, wgt):
    usq = sum(v * v for v in u)
    out = []
    for e, w in zip(vel, wgt):
        cu = sum(k * v for k, v in zip(e, u) if k) if any(e) else torch.zeros_like(rho)
        out.append(w * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * usq))
    return out


def _lbm(fields, steps, tau, vel, wgt):
    dims = len(vel[0])
    f = _equilibrium(fields[0], fields[1:1 + dims], vel, wgt)
    for _ in range(steps):
        rho = sum(f)
        u = [sum(e[a] * g for e, g in zip(vel, f) if e[a]) / rho for a in range(dims)]
        feq = _equilibrium(rho, u, vel, wgt)
        f = [torch.roll(g - (g - q) / tau, tuple(e), tuple(range(dims - 1, -1, -1))) for g, q, e in zip(f, feq, vel)]
    return torch.stack(f)


def _neighbours(W, periodic):
    """W[F, y, x] at x + 1, x - 1, y + 1, y - 1 (wrapped, or the border node copied)."""
    out = []
    for dim, d in ((2, 1), (2, -1), (1, 1), (1, -1)):
        if periodic:
            out.append(torch.roll(W, -d, dim))
            continue
        n = W.shape[dim]
        idx = (torch.arange(n, device=W.device) + d).clamp(0, n - 1)
        out.append(W.index_select(dim, idx))
    return out


_NORMALS = ((1, 0), (-1, 0), (0, 1), (0, -1))


def _euler(c, fields, gamma=1.4):
    rho, u, v, p = fields
    W = torch.stack([rho, rho * u, rho * v, p / (gamma - 1) + 0.5 * rho * (u * u + v * v)])
    t = 0.0

    def prim(W):
        u, v = W[1] / W[0], W[2] / W[0]
        p = (gamma - 1) * (W[3] - 0.5 * (W[1] * u + W[2] * v))
        return u, v, p, torch.sqrt(gamma * p / W[0])

    for _ in range(c["steps"]):
        u, v, p, s = prim(W)
        lam = c["cfl"] / float(torch.maximum(u.abs() + s, v.abs() + s).max()) if c["cfl"] > 0 else -c["cfl"]
        acc = torch.zeros_like(W)
        for N, (a, b) in zip(_neighbours(W, c["periodic"]), _NORMALS):
            un, vn, pn, sn = prim(N)
            q, qn = u * a + v * b, un * a + vn * b
            m = torch.maximum(q.abs() + s, qn.abs() + sn)
            fl = lambda W, q, p: torch.stack([W[0] * q, W[1] * q + p * a, W[2] * q + p * b, (W[3] + p) * q])
            acc += 0.5 * (fl(W, q, p) + fl(N, qn, pn)) - 0.5 * m * (N - W)
        W = W - lam * acc
        t += lam / c["nx"]
    return W, t


def _transport(c, fields, vel):
    W, (a, b) = fields[0][None], vel
    lam = c["cfl"] / max(abs(a), abs(b))
    for _ in range(c["steps"]):
        acc = torch.zeros_like(W)
        for N, aN in zip(_neighbours(W, c["periodic"]), (a, -a, b, -b)):
            acc += W * max(aN, 0.0) + N * min(aN, 0.0)
        W = W - lam * acc
    return W, c["steps"] * lam * 2.0 / c["nx"]


def _swe(c, fields, g=9.81):
    h, u, v = fields
    W, t = torch.stack([h, h * u, h * v]), 0.0

    def fK(h, hK):
        rar = 2 * (torch.sqrt(g * h) - torch.sqrt(g * hK))
        q = torch.sqrt(0.5 * g * (h + hK) / (h * hK))
        shock = (h - hK) * q
        return (torch.where(h <= hK, rar, shock),
                torch.where(h <= hK, torch.sqrt(g / h), q - 0.25 * g * (h - hK) / (h * h * q)))

    def riemann(hL, uL, tL, hR, uR, tR):  # exact wet-bed solution at x / t = 0
        cL, cR = torch.sqrt(g * hL), torch.sqrt(g * hR)
        h = (0.5 * (cL + cR) - 0.25 * (uR - uL)) ** 2 / g
        for _ in range(8):
            fl, dl = fK(h, hL)
            fr, dr = fK(h, hR)
            h = h - (fl + fr + uR - uL) / (dl + dr)
        us = 0.5 * (uL + uR) + 0.5 * (fK(h, hR)[0] - fK(h, hL)[0])
        cs = torch.sqrt(g * h)
        left = us >= 0
        s = torch.where(left, 1.0, -1.0)  # the side of the contact, mirrored to the left
        hK, uK, cK = torch.where(left, hL, hR), torch.where(left, uL, -uR), torch.where(left, cL, cR)
        um = us * s
        sK = uK - cK * torch.sqrt(h * (h + hK) / (2 * hK * hK))
        fan = (uK + 2 * cK) / 3
        outer = torch.where(h > hK, sK >= 0, uK - cK >= 0)
        inner = torch.where(h > hK, sK < 0, um - cs <= 0)
        hh = torch.where(outer, hK, torch.where(inner, h, fan * fan / g))
        uu = torch.where(outer, uK, torch.where(inner, um, fan)) * s
        return hh, uu, torch.where(left, tL, tR)

    for _ in range(c["steps"]):
        u, v = W[1] / W[0], W[2] / W[0]
        s = torch.sqrt(g * W[0])
        lam = c["cfl"] / float(torch.maximum(u.abs() + s, v.abs() + s).max()) if c["cfl"] > 0 else -c["cfl"]
        acc = torch.zeros_like(W)
        for N, (a, b) in zip(_neighbours(W, c["periodic"]), _NORMALS):
            un, vn = N[1] / N[0], N[2] / N[0]
            h, q, w = riemann(W[0], u * a + v * b, v * a - u * b, N[0], un * a + vn * b, vn * a - un * b)
            f0, f1, f2 = h * q, h * q * q + 0.5 * g * h * h, h * q * w
            acc += torch.stack([f0, f1 * a - f2 * b, f1 * b + f2 * a])
        W = W - lam * acc
        t += lam / c["nx"]
    return W, t


def _lift(u, L, dim, inverse=False):
    """Folded BL5/3 lifting of every line of u along one axis of 2^j + 1 nodes."""
    u = u.movedim(dim, 0).contiguous()
    n = u.shape[0] - 1
    for lev in (range(L - 1, -1, -1) if inverse else range(L)):
        s = 1 << lev
        ev, od = u[0:n + 1:2 * s], u[s:n + 1:2 * s]
        a = torch.full((od.shape[0],) + (1,) * (u.dim() - 1), 0.25, dtype=u.dtype, device=u.device)
        a[0] = a[-1] = 0.5
        sign = -1.0 if inverse else 1.0
        for stage in ((1, 0) if inverse else (0, 1)):
            if stage == 0:
                od -= sign * 0.5 * (ev[:-1] + ev[1:])
            else:
                ev[1:-1] += sign * ((a * od)[:-1] + (a * od)[1:])
    return u.movedim(0, dim)


def _labels(c, seed):
    d = _snapshot(c, seed).double()
    P, L, F, dims = c["P"], c["L"], d.shape[0], d.dim() - 1
    E = P + 1
    d = torch.nn.functional.pad(d[None], (0, 1) * dims, mode="circular")[0]
    for ax in range(1, dims + 1):
        d = d.unfold(ax, E, P)
    d = d.reshape(F, -1, *([E] * dims)).transpose(0, 1).contiguous()  # patch, field, nodes
    co = d
    for ax in range(dims, 0, -1):
        co = _lift(co, L, ax + 1)
    co = co.contiguous()
    k = torch.arange(E, device=DEV)
    cls = torch.zeros(E, dtype=torch.long, device=DEV)
    for m in range(L, 0, -1):
        cls = torch.where((k & (1 << (m - 1))) != 0, torch.full_like(cls, m), cls)
    g = torch.meshgrid(*[cls] * dims, indexing="ij")  # slowest axis first
    top = torch.stack(g).amax(0)
    axes = sum(((g[dims - 1 - a] == top).long() << a) for a in range(dims))
    feat = []
    for lev in range(1, L + 1):
        for S in range(1, 1 << dims):
            v = co[:, :, (top == lev) & (axes == S)]
            feat += [torch.log10((v * v).mean((1, 2)) + 1e-30), torch.log10(v.abs().amax((1, 2)) + 1e-30)]
    detail = top > 0
    norm = d.flatten(1).norm(dim=1)

    def err(eps):
        t = torch.where(detail & (co.abs() < eps.reshape(-1, *([1] * (dims + 1)))), 0.0, co)
        for ax in range(1, dims + 1):
            t = _lift(t, L, ax + 1, True)
        return (t - d).flatten(1).norm(dim=1) <= c["delta"] * norm

    best = torch.full((d.shape[0],), -1, dtype=torch.long, device=DEV)
    for q in range(41):
        ok = err(torch.full_like(norm, 10.0 ** (-7 + q / 8)))
        best = torch.where(ok, torch.full_like(best, q), best)
    lo = 10.0 ** (-7 + best.clamp(0, 40).double() / 8)
    hi = 10.0 ** (-7 + (best + 1).clamp(0, 40).double() / 8)
    for _ in range(4):
        mid = torch.sqrt(lo * hi)
        ok = err(mid)
        lo, hi = torch.where(ok, mid, lo), torch.where(ok, hi, mid)
    lab = torch.where(best < 0, -7.0, torch.where(best == 40, -2.0, torch.log10(lo)))
    return {"features": torch.stack(feat, 1), "labels": lab}


def _fit(c, seed, lr=2e-3, sd_floor=1e-3, H=64):
    X, t = (v.double() for v in _samples(c, seed))
    n, nin, nb = c["n"], c["nin"], c["n"] // c["batch"]
    rng = np.random.default_rng(seed)
    W = []
    for i, o in ((nin, H), (H, H), (H, 1)):
        W += [torch.tensor(rng.normal(0, 1 / np.sqrt(i), i * o).astype(np.float32).reshape(o, i)).double().to(DEV),
              torch.zeros(o, dtype=torch.float64, device=DEV)]
    mean, sd = X.mean(0), X.std(0).clamp_min(sd_floor)
    Xs = (X - mean) / sd
    W[5] += t.mean()
    W = [w.requires_grad_() for w in W]
    opt = torch.optim.Adam(W, lr=lr)
    rng = np.random.default_rng(seed)
    hist = []
    for _ in range(c["epochs"]):
        order = torch.tensor(rng.permutation(n)[:nb * c["batch"]], device=DEV)
        for b in order.split(c["batch"]):
            h = torch.nn.functional.gelu(Xs[b] @ W[0].T + W[1])
            h = torch.nn.functional.gelu(h @ W[2].T + W[3])
            loss = (((h @ W[4].T + W[5])[:, 0] - t[b]) ** 2).mean()
            opt.zero_grad()
            loss.backward()
            opt.step()
        hist.append(loss.detach())
    W = [w.detach() for w in W]
    W[0] = W[0] / sd
    W[1] = W[1] - W[0] @ mean
    return {"weights": torch.cat([w.reshape(-1) for w in W]), "loss": torch.stack(hist)}


def exact(case, seed):
    """What run() returns, by the uncompressed scheme in FP64 (runs), or by
    plain FP64 torch (labels, training); bytes have no such value."""
    c = case
    if c["kind"] == "labels":
        return _labels(c, seed)
    if c["kind"] == "fit":
        return _fit(c, seed)
    if c["kind"] == "batch":
        states = []
        for k, n in enumerate(_batch_list(c)):
            one = _run("", "d2q9", n, n, 64, 4, c["eps"], c["steps"], tau=c["tau"], init="bump")
            states.append(_lbm(_fields(one, 1000 * seed + k), c["steps"], c["tau"], *_D2))
        return {"states": states, "bytes": None}
    if c["kind"] != "run":
        return None
    f = _fields(c, seed)
    if c["scheme"] in ("d2q9", "d3q19"):
        W = _lbm(f, c["steps"], c["tau"], *(_D2 if c["scheme"] == "d2q9" else _D3))
        t = float(c["steps"]) if c["scheme"] == "d2q9" else None
    elif c["scheme"] == "euler2d":
        W, t = _euler(c, f)
    elif c["scheme"] == "transport":
        W, t = _transport(c, f, _velocity(seed))
    else:
        W, t = _swe(c, f)
    sums = W
    if not c["periodic"]:  # trapezoid weights on the border nodes
        sums = W.clone()
        for d in (1, 2):
            for k in (0, -1):
                sums.select(d, k).mul_(0.5)
    keep = c["wavelet"] != "cdf97"  # that transform keeps no trapezoid mass
    return {"state": W, "field_sum": sums.flatten(1).sum(1) if keep else None, "time": t, "bytes": None}
