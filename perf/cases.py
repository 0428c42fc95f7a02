"""The work users have this package do, as cases that can be timed.

Kinds of case:

* ``foam``: ``steps`` time steps of a foaming run through ``Sim.step``, then
  the fields a monitoring program keeps (on the device) and the bubble table.
  The lattice starts as liquid below a free surface (or filled, when
  periodic), stirred by a seeded smooth flow where ``stir`` is set, with
  seeded nuclei already carved; a state keeps running when it is run again.
* ``flow``: the same call on a lattice without gas (channel and cavity
  flows, viscometry), any collision model.
* ``label``: bubble labels of a device cell-type field.
* ``forward``, ``generate``, ``train``: the learned curvature on its own --
  a batch of stencils through the network, synthetic training pairs, and a
  training run.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1908_04262_gb300 import lbf as L
from paper_1908_04262_gb300 import workloads as W

FIELDS = ("rho", "u", "alpha", "flags", "conc", "label")


def listed():
    return [
        # one step and a look at the state, the loop of an interactive or
        # coupled program, on the 32^3 crop of the 128^3 workload: latency
        dict(name="crop32_fp32_step1", kind="foam", nx=32, ny=32, nz=32, storage="fp32", rheo="powerlaw", steps=1,
             nuclei=1, rmin=5.0, rmax=5.0, spacing=0.0, walled=True, stir=True, mlp=False, kappa=0),
        # the 2D growth study, 128^2 in double precision
        dict(name="growth2d_128_fp64", kind="foam", nx=128, ny=128, nz=1, storage="fp64", rheo="newtonian", steps=20,
             nuclei=1, rmin=8.0, rmax=8.0, spacing=0.0, walled=True, stir=True, mlp=False, kappa=0),
        # the 2D foam drainage run of Sec. 4.4 at its size, gravity on
        dict(name="drainage2d_450x650_fp32", kind="foam", nx=450, ny=650, nz=1, storage="fp32", rheo="newtonian",
             steps=20, nuclei=150, rmin=3.0, rmax=3.0, spacing=9.0, walled=True, stir=True, mlp=False, kappa=0),
        # one bubble in a periodic box in double precision: the Laplace test
        # and the runs the learned curvature harvests its data from (R = 12)
        dict(name="bubble3d_40_fp64", kind="foam", nx=40, ny=40, nz=40, storage="fp64", rheo="newtonian", steps=20,
             nuclei=1, rmin=12.0, rmax=12.0, spacing=0.0, walled=False, stir=True, mlp=False, kappa=0),
        # the headline workload: 128^3, FP32, power law, 8 bubbles
        dict(name="foam3d_128_fp32", kind="foam", nx=128, ny=128, nz=128, storage="fp32", rheo="powerlaw", steps=20,
             nuclei=8, rmin=4.0, rmax=6.0, spacing=20.0, walled=True, stir=True, mlp=False, kappa=0),
        # its second form: shifted FP16 storage and the learned curvature
        dict(name="foam3d_128_fp16s_mlp", kind="foam", nx=128, ny=128, nz=128, storage="fp16s", rheo="powerlaw",
             steps=20, nuclei=8, rmin=4.0, rmax=6.0, spacing=20.0, walled=True, stir=True, mlp=True, kappa=0),
        # the 256^3 Carreau foam with its 200 nuclei, shifted FP16
        dict(name="foam3d_256_fp16s", kind="foam", nx=256, ny=256, nz=256, storage="fp16s", rheo="carreau", steps=8,
             nuclei=200, rmin=2.0, rmax=4.0, spacing=8.0, walled=True, stir=True, mlp=False, kappa=0),
        # the largest run: 100 million cells, 2000 nuclei, shifted BF16, the
        # learned curvature; its monitor keeps fill levels and bubble
        # statistics (the flow starts at rest)
        dict(name="foam3d_512x512x384_bf16s", kind="foam", nx=512, ny=512, nz=384, storage="bf16s", rheo="powerlaw",
             steps=4, nuclei=2000, rmin=2.0, rmax=4.0, spacing=10.0, walled=True, stir=False, mlp=True, kappa=0),
        # a forced power-law flow without gas on a ragged periodic lattice,
        # two relaxation times
        dict(name="flow3d_201x77x131_fp32", kind="flow", nx=201, ny=77, nz=131, storage="fp32", rheo="powerlaw",
             collision=1, walled=False, steps=20),
        # bubble labels for a program that may not allocate
        dict(name="label_101x96x99", kind="label", nx=101, ny=96, nz=99, bubbles=60, rmin=3.0, rmax=9.0),
        # the network over the interface cells of a large foam
        dict(name="mlp_forward_503117", kind="forward", n=503117),
        # a training run: generated stencils, mini-batches of 2048, Adam
        dict(name="mlp_train_98304", kind="train", n=98304, epochs=1, batch=2048),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["foam3d"] * 4 + ["foam2d"] * 2 + ["flow"] * 2 + ["label", "forward", "generate", "train"])
    if kind == "foam2d":
        nx, ny = (int(_log(rng, 48, 1000)) for _ in range(2))
        return dict(kind="foam", nx=nx, ny=ny, nz=1, storage=rng.choice(["fp64", "fp32", "fp32", "fp16s"]),
                    rheo="newtonian", steps=rng.choice([1, 4, 13, 20]), nuclei=max(1, nx * ny // 3000), rmin=3.0,
                    rmax=5.0, spacing=13.0, walled=rng.random() < 0.8, stir=True, mlp=False,
                    kappa=int(rng.random() < 0.25))
    if kind == "foam3d":
        nx, ny, nz = (int(_log(rng, 32, 230)) for _ in range(3))
        storage = rng.choice(["fp32", "fp32", "fp16s", "bf16s", "fp64"])
        if storage == "fp64":
            nx, ny, nz = min(nx, 90), min(ny, 90), min(nz, 90)
        return dict(kind="foam", nx=nx, ny=ny, nz=nz, storage=storage,
                    rheo=rng.choice(["newtonian", "powerlaw", "carreau"]), steps=rng.choice([1, 4, 9, 16]),
                    nuclei=max(1, nx * ny * nz // 100000), rmin=3.0, rmax=5.0, spacing=12.0,
                    walled=rng.random() < 0.8, stir=True, mlp=rng.random() < 0.3, kappa=int(rng.random() < 0.2))
    if kind == "flow":
        flat = rng.random() < 0.3
        nx, ny, nz = (int(_log(rng, 40, 1500 if flat else 220)) for _ in range(3))
        return dict(kind="flow", nx=nx, ny=ny, nz=1 if flat else nz, storage=rng.choice(["fp32", "fp32", "fp64"]),
                    rheo=rng.choice(["newtonian", "powerlaw"]), collision=rng.choice([0, 1]),
                    walled=rng.random() < 0.5, steps=rng.choice([4, 9, 20]))
    if kind == "label":
        return dict(kind="label", nx=rng.randint(20, 128), ny=rng.randint(20, 90), nz=rng.choice([1, rng.randint(20, 90)]),
                    bubbles=rng.randint(5, 120), rmin=2.0, rmax=9.0)
    if kind == "forward":
        return dict(kind="forward", n=int(_log(rng, 200, 2000000)))
    if kind == "generate":
        return dict(kind="generate", n=int(_log(rng, 1000, 400000)))
    batch = rng.choice([512, 2048, 4099])
    return dict(kind="train", n=batch * rng.randint(4, 24) + rng.randint(0, 300), epochs=1, batch=batch)


# ---------------------------------------------------------------------------
# inputs


def _config(c):
    """The physics of the package's workload of the same kind on this lattice."""
    base = dict(nx=c["nx"], ny=c["ny"], nz=c["nz"], storage=c["storage"], collision=c.get("collision", 0),
                kappa=c.get("kappa", 0))
    flat = c["nz"] == 1
    n_up = c["ny"] if flat else c["nz"]
    base["walls"] = (0xF if flat else 0x3F) if c["walled"] else 0
    if c["kind"] == "flow":
        base.update(atmosphere=0, tau=0.8, accel=(2e-5, 0.0, 0.0), D=0.03, c0=1.0)
    elif not c["walled"]:
        base.update(atmosphere=0, tau=0.8, sigma=0.01, kH=0.0, D=0.05, c0=0.0, p0=1.0 / 3.0)
    elif flat and c["nuclei"] == 1:
        base.update(tau=0.8, sigma=0.01, D=0.05, kH=0.5, c0=1.0, RT=0.1, fill_height=0.875 * n_up)
    elif flat:
        base.update(tau=0.95, sigma=5e-3, k_pi=2e-3, d_max=3.0, D=0.01, kH=1e-5, c0=0.02, RT=5.0,
                    accel=(0.0, -3e-5, 0.0), fill_height=0.6 * n_up)
    else:
        base.update(tau=0.7, sigma=5e-3, d_max=3.0, k_pi=1e-3 / 3.0, D=0.02, kH=0.5, c0=1.0, RT=0.1,
                    fill_height=0.75 * n_up)
    if c["rheo"] == "powerlaw":
        n = 0.6
        base.update(rheo=W.RHEO["powerlaw"], rheo_n=n, rheo_k=W.powerlaw_k(n))
    elif c["rheo"] == "carreau":
        base.update(rheo=W.RHEO["carreau"], rheo_n=0.5, rheo_lambda=50.0, rheo_a=2.0, tau0=0.8, tau_inf=0.505, tau=0.8)
    return W.config(**base)


def _stirred(cfg, rng):
    """Cell arrays of the initial fill with a smooth flow of amplitude 0.02."""
    nx, ny, nz = cfg["nx"], cfg["ny"], cfg["nz"]
    flat = nz == 1
    ax = [np.arange(n, dtype=np.float64) for n in (nx, ny, nz)]

    def mode(d):
        k, ph = rng.integers(1, 4), rng.uniform(0, 2 * np.pi)
        shape = [1, 1, 1]
        shape[2 - d] = -1
        return np.sin(2 * np.pi * k * ax[d] / len(ax[d]) + ph).reshape(shape)

    u = np.zeros((nz, ny, nx, 3))
    amp = 0.02
    u[..., 0] = amp * mode(1) * (1.0 if flat else mode(2))
    u[..., 1] = amp * mode(0) * (1.0 if flat else mode(2))
    if not flat:
        u[..., 2] = amp * mode(0) * mode(1)
    up = ax[1] if flat else ax[2]
    fill = np.clip(cfg["fill_height"] - (up - 0.5), 0.0, 1.0).reshape((1, -1, 1) if flat else (-1, 1, 1))
    alpha = np.broadcast_to(fill, (nz, ny, nx)).copy()
    types = np.where(alpha >= 1.0, 1, np.where(alpha <= 0.0, 0, 2)).astype(np.uint8)
    for bit, face in enumerate((np.s_[:, :, 0], np.s_[:, :, -1], np.s_[:, 0], np.s_[:, -1], np.s_[0], np.s_[-1])):
        if cfg["walls"] >> bit & 1 and not (flat and bit > 3):
            types[face] = 3
    rho = np.full(nx * ny * nz, cfg["rho0"])
    conc = np.full(nx * ny * nz, cfg["c0"])
    return types.reshape(-1), rho, u.reshape(-1, 3), alpha.reshape(-1), conc


def _nuclei(c, cfg, rng):
    """Seeded sites in the liquid, at least ``spacing`` apart and clear of the faces."""
    flat = c["nz"] == 1
    n_up = min(cfg["fill_height"], c["ny"] if flat else c["nz"])
    hi = np.array([c["nx"] - 3.0, n_up - 5.0] if flat else [c["nx"] - 3.0, c["ny"] - 3.0, n_up - 5.0])
    lo = np.full(len(hi), 2.0)
    if c["nuclei"] == 1:
        r = np.array([min(c["rmax"], 0.5 * float(np.min(hi - lo)) - 3.0)])
        pts = (lo + hi)[None, :] / 2 + rng.uniform(-0.5, 0.5, (1, len(hi)))
    else:
        size = c["nuclei"]
        while True:
            try:
                pts, r = W.poisson_disk(rng, size, lo, hi, c["spacing"], c["rmin"], c["rmax"], max_tries=20 * size)
                break
            except RuntimeError:
                size = max(1, size // 2)
    return W.as3(pts), r


def _sphere_stencils(n, gen, dev):
    """Canonically oriented 3x3x3 fill levels of spheres (gas inside, radii
    log-uniform in [2, 40]) around a surface cell, and 4 / R, in FP64."""
    rnd = lambda *s: torch.rand(*s, generator=gen, dtype=torch.float64, device=dev)  # noqa: E731
    R = torch.exp(math.log(2.0) + rnd(n) * math.log(20.0))
    d = torch.sort(torch.abs(torch.randn(n, 3, generator=gen, dtype=torch.float64, device=dev)), dim=1)[0]
    d = d / d.norm(dim=1, keepdim=True)
    centre = -d * (R + rnd(n) - 0.5)[:, None]
    x = torch.zeros(n, 27, dtype=torch.float64, device=dev)
    sub = [(k + 0.5) / 3 - 0.5 for k in range(3)]
    q = torch.arange(27, device=dev)
    off = torch.stack([q % 3 - 1, (q // 3) % 3 - 1, q // 9 - 1], 1).double()
    for sx in sub:
        for sy in sub:
            for sz in sub:
                d2 = 0
                for a, s in enumerate((sx, sy, sz)):
                    d2 = d2 + (off[None, :, a] + s - centre[:, None, a]) ** 2
                x += (d2 >= (R * R)[:, None]).double()
    return x / 27, 4.0 / R


def _network(rng):
    """Seeded random parameters of the curvature network (6017 float32)."""
    parts = [rng.normal(0, 27 ** -0.5, 64 * 27), rng.normal(0, 0.1, 64), rng.normal(0, 64 ** -0.5, 64 * 64),
             rng.normal(0, 0.1, 64), rng.normal(0, 64 ** -0.5, 64), np.zeros(1)]
    return np.concatenate(parts).astype(np.float32)


def _fitted_network(seed):
    """Random hidden layers and an output layer fitted to sphere stencils:
    a network whose curvature is about right, made in a moment."""
    th = _network(np.random.default_rng(seed)).astype(np.float64)
    gen = torch.Generator().manual_seed(seed)
    x, y = (t.numpy() for t in _sphere_stencils(1500, gen, "cpu"))
    silu = lambda z: z / (1 + np.exp(-z))  # noqa: E731
    h = silu(x @ th[:1728].reshape(64, 27).T + th[1728:1792])
    h = silu(h @ th[1792:5888].reshape(64, 64).T + th[5888:5952])
    h = np.concatenate([h, np.ones((len(h), 1))], 1)
    th[5952:] = np.linalg.solve(h.T @ h + 1e-3 * len(h) * np.eye(65), h.T @ y)
    return th.astype(np.float32)


def _flow_state(cfg, seed):
    """Cell types, density, velocity (a smooth flow of amplitude 0.05 with
    seeded perturbations of every cell) and dissolved gas."""
    types, _, smooth, _, _ = _stirred(cfg, np.random.default_rng(seed))
    rho, noise, conc = W.random_flow_state(cfg, seed)
    return types, rho, 2.5 * smooth + noise, conc


def prepare(c, seed):
    kind = c["kind"]
    rng = np.random.default_rng(seed)
    if kind in ("foam", "flow"):
        cfg = _config(c)
        stream = torch.cuda.Stream()
        sim = L.Sim(cfg, stream=stream.cuda_stream)
        N = sim.N
        if kind == "flow":
            types, rho, u, conc = _flow_state(cfg, seed)
            sim.set_cells(types, rho, u, np.ones(N), conc)
        else:
            if c["stir"]:
                sim.set_cells(*_stirred(cfg, rng))
            sim.nucleate(*_nuclei(c, cfg, rng))
            if c["mlp"]:
                sim.mlp_attach(_fitted_network(seed))
        real = torch.float64 if c["storage"] == "fp64" else torch.float32
        keep = ("rho", "u", "conc") if kind == "flow" else (FIELDS if c["stir"] else tuple(f for f in FIELDS if f != "u"))
        out = {}
        for k in keep:
            shape = (N, 3) if k in L.VECTOR_FIELDS else (N,)
            out[k] = torch.empty(shape, dtype=torch.int32 if k in L.INT_FIELDS else real, device="cuda")
        torch.cuda.synchronize()
        return dict(c, sim=sim, stream=stream, out=out)
    if kind == "label":
        nx, ny, nz = c["nx"], c["ny"], c["nz"]
        gen = torch.Generator(device="cuda").manual_seed(seed)
        ctr = torch.rand(c["bubbles"], 3, generator=gen, device="cuda") * torch.tensor([nx, ny, nz], device="cuda")
        rad = c["rmin"] + (c["rmax"] - c["rmin"]) * torch.rand(c["bubbles"], generator=gen, device="cuda")
        z, y, x = torch.meshgrid(*(torch.arange(n, device="cuda", dtype=torch.float32) for n in (nz, ny, nx)), indexing="ij")
        d = torch.full((nz, ny, nx), 1e9, device="cuda")  # distance to the nearest surface
        for i in range(c["bubbles"]):
            r2 = (x - ctr[i, 0]) ** 2 + (y - ctr[i, 1]) ** 2 + ((z - ctr[i, 2]) ** 2 if nz > 1 else 0)
            d = torch.minimum(d, r2.sqrt() - rad[i])
        types = torch.where(d < 0, 0, torch.where(d < 1.5, 2, 1)).to(torch.uint8).reshape(-1)
        N = nx * ny * nz
        s = dict(c, types=types, labels=torch.empty(N, dtype=torch.int32, device="cuda"),
                 count=torch.zeros(1, dtype=torch.int32, device="cuda"))
        return s
    if kind == "forward":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x = _sphere_stencils(c["n"], gen, "cuda")[0].float()
        return dict(c, theta=torch.tensor(_network(rng), device="cuda"), x=x,
                    y=torch.empty(c["n"], device="cuda"))
    if kind == "generate":
        return dict(c, seed=seed, x=torch.empty(c["n"], 27, device="cuda"), y=torch.empty(c["n"], device="cuda"))
    return dict(c, seed=seed, theta=_network(rng))


def run(s):
    kind = s["kind"]
    if kind in ("foam", "flow"):
        sim = s["sim"]
        sim.step(s["steps"])
        sim.fields_device(s["out"], 1 if s["storage"] == "fp64" else 0)
        b = sim.bubbles()  # waits for the stream: the fields are written too
        if kind == "flow":
            return s["out"]
        # the table is kept in the run's arithmetic precision
        real = np.float64 if s["storage"] == "fp64" else np.float32
        return dict(s["out"], table={k: v.astype(real) if v.dtype.kind == "f" else v for k, v in b.items()})
    if kind == "label":
        L.label_gas_noalloc(s["types"], s["nx"], s["ny"], s["nz"], s["labels"], s["count"])
        return s["labels"], s["count"]
    if kind == "forward":
        L.mlp_forward(s["theta"], s["x"], s["y"])
        return s["y"]
    if kind == "generate":
        L.mlp_generate(s["seed"], s["x"], s["y"])
        return s["x"], s["y"]
    return L.mlp_train(s["theta"], n_samples=s["n"], epochs=s["epochs"], batch=s["batch"], seed=s["seed"])


def work(c):
    kind = c["kind"]
    if kind in ("foam", "flow"):
        flat = c["nz"] == 1
        N, Q = c["nx"] * c["ny"] * c["nz"], 14 if flat else 26
        size = {"fp64": 8, "fp32": 4}.get(c["storage"], 2)
        real = 8 if c["storage"] == "fp64" else 4
        if kind == "flow":
            fluid, ifc = N, 0
        else:
            cfg = _config(c)
            n_up = c["ny"] if flat else c["nz"]
            fluid = int(N * min(1.0, cfg["fill_height"] / n_up))
            rm = 0.5 * (c["rmin"] + c["rmax"])
            # a shell of a cell and a half around each bubble, and the free surface
            ifc = c["nuclei"] * 1.5 * (2 * math.pi * rm if flat else 4 * math.pi * rm * rm)
            ifc = int(ifc + (N // n_up if c["walled"] else 0))
        gas = N - fluid
        # each step: every population of a fluid cell in and out once and its
        # flag; an interface cell's mass, fill level, velocity, curvature,
        # normal and pressures; a gas cell's flag and label
        step = fluid * (2 * Q * size + 2) + ifc * 30 * real + gas * 9
        per = 3 if kind == "flow" else 4
        look = fluid * Q * size + N * (per * real + (0 if kind == "flow" else 8) + (3 * real if c.get("stir", True) else 0))
        return {"bytes": c["steps"] * step + look, "flops": c["steps"] * fluid * Q * 14.0}
    if kind == "label":
        N = c["nx"] * c["ny"] * c["nz"]
        return {"bytes": N * 5, "flops": 0}
    net = 2.0 * (27 * 64 + 64 * 64 + 64)
    if kind == "forward":
        return {"bytes": c["n"] * 28 * 4 + 6017 * 4, "flops": c["n"] * net}
    if kind == "generate":
        return {"bytes": c["n"] * 28 * 4, "flops": c["n"] * 27 * 216 * 15.0}
    seen = c["epochs"] * (c["n"] // c["batch"]) * c["batch"]
    # stencils are made once, read once an epoch; forward, both backward products
    return {"bytes": c["n"] * 28 * 4 + seen * 28 * 4 + 6017 * 4 * 8, "flops": c["n"] * 27 * 216 * 15.0 + 3 * seen * net}


# ---------------------------------------------------------------------------
# the same in 64 bits, without this package's kernels


def _lattice(flat):
    e = [(0, 0, 0)]
    if flat:
        half = [(1, 0, 0), (0, 1, 0), (1, 1, 0), (1, -1, 0)]
        w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
    else:
        half = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, 0, 1), (0, 1, 1), (1, -1, 0), (1, 0, -1), (0, 1, -1)]
        w = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
    for v in half:
        e += [v, tuple(-a for a in v)]
    qa = 5 if flat else 7
    wa = [1 / 3] + [1 / 6] * 4 if flat else [1 / 4] + [1 / 8] * 6
    return e, w, qa, wa, (1 / 3 if flat else 1 / 4)


def _exact_flow(c, seed):
    cfg = _config(c)
    flat = c["nz"] == 1
    e, w, qa, wa, ca2 = _lattice(flat)
    shape = (c["nz"], c["ny"], c["nx"])
    types, r0, u0, c0 = _flow_state(cfg, seed)
    wall = torch.tensor(types.reshape(shape) == 3, device="cuda")
    rho = torch.tensor(r0.reshape(shape), device="cuda")
    u = [torch.tensor(np.ascontiguousarray(u0[:, d]).reshape(shape), device="cuda") for d in range(3)]
    conc = torch.tensor(c0.reshape(shape), device="cuda")
    a = cfg["accel"]
    dot = lambda v, x: sum(k * x[d] for d, k in enumerate(v) if k) if any(v) else torch.zeros_like(rho)  # noqa: E731

    def feq(i, rho, u):
        eu, uu = dot(e[i], u), u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        return w[i] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * uu)

    f = [feq(i, rho, u) for i in range(len(e))]
    g = [wa[i] * conc * (1 + dot(e[i], u) / ca2) for i in range(qa)]

    def stream(p):
        # an own outgoing population that would come from a wall is reflected
        opp = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, len(p))]
        out = []
        for i in range(len(p)):
            sh = (e[i][2], e[i][1], e[i][0])
            got = torch.roll(p[i], sh, (0, 1, 2))
            from_wall = torch.roll(wall, sh, (0, 1, 2))
            out.append(torch.where(from_wall, p[opp[i]], got))
        return out

    for _ in range(c["steps"]):
        f, g = stream(f), stream(g)
        rho = sum(f)
        rho = torch.where(wall, torch.ones_like(rho), rho)
        u = [sum(f[i] * e[i][d] for i in range(len(e)) if e[i][d]) if any(v[d] for v in e) else torch.zeros_like(rho)
             for d in range(3)]
        u = [(u[d] + 0.5 * rho * a[d]) / rho for d in range(3)]
        tau = torch.full_like(rho, cfg["tau"])
        if cfg["rheo"]:
            neq = torch.zeros_like(rho)
            for p in range(3):
                for q in range(3):
                    m = sum((f[i] * (e[i][p] * e[i][q]) for i in range(len(e)) if e[i][p] * e[i][q]), torch.zeros_like(rho))
                    m = m - rho * u[p] * u[q]
                    if p == q and not (flat and p == 2):
                        m = m - rho / 3
                    neq += m * m
            A = neq.sqrt() * (3 / math.sqrt(2.0)) / rho
            lo, hi = torch.full_like(rho, cfg["tau_min"]), torch.full_like(rho, cfg["tau_max"])
            for _ in range(60):
                mid = 0.5 * (lo + hi)
                model = 0.5 + 3 * cfg["rheo_k"] * (A / mid) ** (cfg["rheo_n"] - 1)
                up = mid > model
                hi, lo = torch.where(up, mid, hi), torch.where(up, lo, mid)
            tau = 0.5 * (lo + hi)
        om = 1 / tau
        om_m = 1 / (0.5 + cfg["trt_magic"] / (tau - 0.5)) if c["collision"] == 1 else om
        new = []
        for i in range(len(e)):
            j = 0 if i == 0 else (i + 1 if i % 2 else i - 1)
            fi, fj = feq(i, rho, u), feq(j, rho, u)
            F = [w[k] * rho * (3 * (dot(e[k], a) if any(e[k]) else 0.0) - 3 * dot(a, u) + 9 * dot(e[k], u) * (sum(x * y for x, y in zip(e[k], a))))
                 for k in (i, j)]
            even, odd = 0.5 * (f[i] + f[j]), 0.5 * (f[i] - f[j])
            even = even - (even - 0.5 * (fi + fj)) * om + (1 - 0.5 * om) * 0.5 * (F[0] + F[1])
            odd = odd - (odd - 0.5 * (fi - fj)) * om_m + (1 - 0.5 * om_m) * 0.5 * (F[0] - F[1])
            new.append(even + odd)
        f = new
        cg = sum(g)
        omg = 1 / (0.5 + cfg["D"] / ca2)
        g = [g[i] + (wa[i] * cg * (1 + dot(e[i], u) / ca2) - g[i]) * omg for i in range(qa)]
    rho = sum(f)
    rho = torch.where(wall, torch.ones_like(rho), rho)
    u = torch.stack([(sum((f[i] * e[i][d] for i in range(len(e)) if e[i][d]), torch.zeros_like(rho)) - 0.5 * rho * a[d]) / rho
                     for d in range(3)], -1)
    fluid = ~wall
    return {"rho": (rho * fluid).reshape(-1), "u": (u * fluid[..., None]).reshape(-1, 3), "conc": (sum(g) * fluid).reshape(-1)}


def exact(c, seed):
    kind = c["kind"]
    if kind == "flow":
        return _exact_flow(c, seed)
    if kind == "forward":
        s = prepare(c, seed)
        th, y = s["theta"].double(), []
        for x in s["x"].double().split(1 << 18):
            h = torch.nn.functional.silu(x @ th[:1728].view(64, 27).T + th[1728:1792])
            h = torch.nn.functional.silu(h @ th[1792:5888].view(64, 64).T + th[5888:5952])
            y.append(h @ th[5952:6016] + th[6016])
        return torch.cat(y)
    # a foam's interface moves by rules of its own (no closed form); labels
    # are whole numbers; the training pairs' generator is part of the package
    return None
