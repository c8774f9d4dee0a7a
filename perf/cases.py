"""The calls that users of this library have it do, as measurable cases: moment propagation
(both schemes, all storage types, one context or a group), the lattice-Boltzmann flow solve,
the learned warm start and its training, and the allocation-free step, each through the
public entry points (`mp`, `surrogate`) and with inputs of the kind the repository's own
benchmark, tests and validation runs use.

listed() and draw() give cases, prepare() their inputs and handles, run() one pass, work()
what a pass cannot do without, and exact() the same results in 64 bits from plain torch.
"""
import math

import numpy as np
import torch

# ------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------


def listed():
    return [
        # the paper's slit pore (D(t) normal to the walls), FP64 fields, one small context of
        # its own: many thousand launches of a few hundred nodes
        {"name": "slit_fp64", "kind": "slit", "width": 3, "L": 100, "species": 1, "flow": False, "steps": 4096},
        # the paper's periodic fcc packing at its full size, four adsorbed fractions in one
        # context, FP32, fluid at rest, default options
        {"name": "fcc100_flux", "kind": "flux", "medium": "fcc", "nx": 100, "ny": 100, "nz": 100, "species": 4,
         "precision": "fp32", "directions": "x", "steps": 600},
        # binary16 field storage (the capacity option) on an uneven porous box, two moments
        {"name": "porous_fp16", "kind": "flux", "medium": "spheres", "nx": 90, "ny": 77, "nz": 101, "species": 1,
         "precision": "fp16", "directions": "xz", "steps": 1000},
        # the benchmark job's propagation: one species on a 128^3 random-sphere medium
        {"name": "direct_128", "kind": "direct", "nx": 128, "ny": 128, "nz": 128, "species": 1, "directions": "x",
         "steps": 2000},
        # several species on a medium whose working set is far beyond L2
        {"name": "direct_256x4", "kind": "direct", "nx": 256, "ny": 256, "nz": 256, "species": 4, "directions": "x",
         "steps": 100},
        # three small media of 16 species each advanced together (a parameter study)
        {"name": "group_16sp", "kind": "group", "n0": 48, "n1": 64, "n2": 80, "species": 16, "steps": 200},
        # a steady flow of the size and force the training set is made of, from rest to 1e-7
        {"name": "lb_64", "kind": "lb", "nx": 64, "ny": 64, "nz": 64, "radius": 6, "porosity": 0.45, "force": 1e-5},
        # the largest flow solve of the batched workload, at a mean velocity of about 0.01
        {"name": "lb_192", "kind": "lb", "nx": 192, "ny": 192, "nz": 192, "radius": 6, "porosity": 0.4,
         "force": 1.8e-3},
        # one step on caller-owned arrays inside another program: the smallest call
        {"name": "noalloc_64", "kind": "noalloc", "nx": 64, "ny": 64, "nz": 64, "direction": 0},
        # warm start of a flow solve from a host mask: node classes, the network, (u, rho)
        {"name": "warm_start_128", "kind": "warm", "nx": 128, "ny": 128, "nz": 128, "axis": 0},
        # one training pass of the network on a batch of 64^3 media: loss and all gradients
        {"name": "train_64x4", "kind": "train", "n": 64, "batch": 4},
        # one convolution layer alone, forward and backward, on an uneven box
        {"name": "layer_uneven", "kind": "layer", "B": 2, "D": 40, "H": 56, "W": 72, "cin": 64, "cout": 64},
    ]


_CHANNELS = [(16, 32), (32, 32), (32, 64), (64, 64), (64, 96), (96, 96), (96, 128), (128, 128), (128, 96),
             (96, 64), (64, 32), (32, 16)]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(lo, hi, cap):
        while True:
            d = [log(lo, hi) for _ in range(3)]
            if d[0] * d[1] * d[2] <= cap:
                return {"nx": d[0], "ny": d[1], "nz": d[2]}

    kind = rng.choice(["slit", "flux", "flux", "direct", "direct", "group", "lb", "noalloc", "warm", "train", "layer",
                       "layer"])
    if kind == "slit":
        c = {"kind": kind, "width": rng.randint(3, 6), "L": log(20, 200), "species": rng.randint(1, 3),
             "flow": rng.random() < 0.5}
        c["steps"] = min(log(1024, 4096), 16_000_000 // (c["width"] ** 2 * (c["L"] + 2) * c["species"]))
        return c
    if kind == "flux":
        c = {"kind": kind, "medium": "spheres", **box(24, 128, 1_000_000), "species": log(1, 8),
             "precision": rng.choice(["fp32", "fp32", "fp16"]), "directions": rng.choice(["x", "xz", "xyz"])}
        c["steps"] = min(1000, max(50, 150_000_000 // (c["nx"] * c["ny"] * c["nz"] * c["species"])))
        return c
    if kind == "direct":
        c = {"kind": kind, **box(32, 256, 8_000_000), "species": log(1, 16),
             "directions": rng.choice(["x", "x", "xz"])}
        c["steps"] = min(1000, max(20, 1_000_000_000 // (c["nx"] * c["ny"] * c["nz"] * c["species"])))
        return c
    if kind == "group":
        return {"kind": kind, "n0": rng.randint(24, 48), "n1": rng.randint(32, 64), "n2": rng.randint(40, 80),
                "species": log(1, 16), "steps": rng.randint(100, 200)}
    if kind == "lb":
        return {"kind": kind, **box(24, 128, 1_000_000), "radius": rng.randint(4, 8),
                "porosity": round(rng.uniform(0.35, 0.6), 3), "force": 10.0 ** round(rng.uniform(-5.0, -3.0), 2)}
    if kind == "noalloc":
        return {"kind": kind, **box(8, 128, 2_000_000), "direction": rng.choice([-1, 0, 1, 2])}
    if kind == "warm":
        return {"kind": kind, "nx": 8 * rng.randint(2, 16), "ny": 8 * rng.randint(2, 16), "nz": 8 * rng.randint(2, 16),
                "axis": rng.randint(0, 2)}
    if kind == "train":
        return {"kind": kind, "n": 8 * rng.randint(3, 8), "batch": rng.randint(1, 4)}
    cin, cout = rng.choice(_CHANNELS)
    while True:
        c = {"kind": "layer", "B": rng.randint(1, 4), "D": log(4, 64), "H": log(4, 64), "W": log(4, 128), "cin": cin,
             "cout": cout}
        if c["B"] * c["D"] * c["H"] * c["W"] <= 400_000:
            return c


# ------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _spheres(nx, ny, nz, radius, porosity, gen):
    """A periodic random-sphere medium on the device, uint8 (nz, ny, nx), 1 = solid: as many
    uniformly placed spheres as give the porosity on average (at least one)."""
    r = int(radius)
    o = torch.arange(-r, r + 1, device="cuda")
    oz, oy, ox = torch.meshgrid(o, o, o, indexing="ij")
    ball = (ox * ox + oy * oy + oz * oz).reshape(-1) <= r * r
    ox, oy, oz = (t.reshape(-1)[ball] for t in (ox, oy, oz))
    n = max(1, int(round(-math.log(porosity) * nx * ny * nz / ox.numel())))
    c = [torch.randint(0, d, (n, 1), generator=gen, device="cuda") for d in (nx, ny, nz)]
    at = (((c[2] + oz) % nz) * ny + (c[1] + oy) % ny) * nx + (c[0] + ox) % nx
    solid = torch.zeros(nx * ny * nz, dtype=torch.uint8, device="cuda")
    solid[at.reshape(-1)] = 1
    solid[0] = 0  # at least one fluid node
    return solid.view(nz, ny, nx)


def _drift(solid, gen):
    """A drift of 0.01 along x with uniform noise of 0.01 on the fluid, FP32 (3, nz, ny, nx)."""
    u = (torch.rand((3,) + tuple(solid.shape), generator=gen, device="cuda") * 2 - 1) * 0.01
    u[0] += 0.01
    u *= (solid == 0)
    return u.contiguous()


def _species(n, rng):
    """D_b in [0.03, 0.1], k_a and k_d log-uniform in [1e-3, 1e-1]."""
    Db = rng.uniform(0.03, 0.1, n)
    ka, kd = (np.exp(rng.uniform(math.log(1e-3), math.log(1e-1), n)) for _ in range(2))
    return Db, ka, kd


def _mp_inputs(case, seed):
    """(solid, u or None, D_b, k_a, k_d) of a moment-propagation case."""
    from paper_1303_2470_gb300 import media, validation
    rng = np.random.default_rng(seed)
    if case["kind"] == "slit":
        w, L, S = case["width"], case["L"], case["species"]
        solid = media.slit(w, w, L)
        ka = np.exp(rng.uniform(math.log(1e-3), math.log(1e-1), S))
        kd = np.exp(rng.uniform(math.log(1e-3), math.log(1e-1), S))
        u = None
        if case["flow"]:
            umax = validation.poiseuille_u_max(L, 0.01, rng.uniform(5.0, 10.0))
            u = torch.as_tensor(media.slit_flow(w, w, L, umax).astype(np.float32)).cuda()
        return solid, u, np.full(S, 0.01), ka, kd
    if case.get("medium") == "fcc":
        solid = media.fcc(case["nx"])
        pairs = np.array(validation.fcc_sorption_pairs(solid, rng.uniform(0.2, 0.97, case["species"])))
        return solid, None, np.full(len(pairs), 0.01), pairs[:, 0].copy(), pairs[:, 1].copy()
    g = _gen(seed)
    solid = _spheres(case["nx"], case["ny"], case["nz"], 6, 0.4, g)
    return (solid, _drift(solid, g)) + _species(case["species"], rng)


def prepare(case, seed):
    from paper_1303_2470_gb300 import mp
    kind = case["kind"]
    s = {"case": case, "kind": kind}
    if kind in ("slit", "flux"):
        s["solid"], s["u"], s["Db"], s["ka"], s["kd"] = _mp_inputs(case, seed)
        s["stream"] = torch.cuda.Stream() if kind == "slit" else None
        torch.cuda.synchronize()
    elif kind == "direct":
        # the program keeps the context (a job is 2e4 steps, in runs between readings of D(t))
        solid, u, Db, ka, kd = _mp_inputs(case, seed)
        s["stream"] = torch.cuda.Stream()
        torch.cuda.synchronize()
        s["ctx"] = mp.mp_init_batch(solid, u, Db, ka, kd, scheme="direct", autotune=True, stream=s["stream"],
                                    directions=case["directions"],
                                    capacity=2_000_000 if case["species"] == 1 else 1_000_000)
    elif kind == "group":
        s["ctxs"] = []
        for k in range(3):
            n = case["n%d" % k]
            solid, u, Db, ka, kd = _mp_inputs({"kind": "group", "nx": n, "ny": n, "nz": n, "species": case["species"]},
                                              seed * 3 + k)
            torch.cuda.synchronize()
            s["ctxs"].append(mp.mp_init_batch(solid, u, Db, ka, kd, scheme="direct", capacity=400_000))
        s["group"] = mp.mp_group_create(s["ctxs"], graph_steps=64, autotune=True)
    elif kind == "lb":
        g = _gen(seed)
        s["solid"] = _spheres(case["nx"], case["ny"], case["nz"], case["radius"], case["porosity"], g)
        s["u"] = torch.zeros((3,) + tuple(s["solid"].shape), device="cuda")
        s["rho"] = torch.zeros(tuple(s["solid"].shape), device="cuda")
    elif kind == "noalloc":
        g = _gen(seed)
        solid = _spheres(case["nx"], case["ny"], case["nz"], 6, 0.4, g)
        s["solid"], s["u"] = solid, _drift(solid, g)
        fluid = (solid == 0)
        s["X"] = torch.rand(solid.shape, generator=g, device="cuda") * fluid
        s["Xa"] = torch.rand(solid.shape, generator=g, device="cuda") * fluid
        s["Xn"], s["Xan"] = torch.empty_like(s["X"]), torch.empty_like(s["X"])
        s["Z"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    elif kind == "warm":
        from paper_1303_2470_gb300 import surrogate
        s["solid"] = _spheres(case["nx"], case["ny"], case["nz"], 6, 0.4, _gen(seed)).cpu().numpy()
        s["model"] = surrogate.load()[0]
        force = [0.0, 0.0, 0.0]
        force[case["axis"]] = 1e-3
        s["force"] = tuple(force)
    elif kind == "train":
        from paper_1303_2470_gb300 import surrogate
        n, B = case["n"], case["batch"]
        g = _gen(seed)
        s["model"] = surrogate.load()[0]
        s["x"], s["t"] = _train_batch(n, B, g)
        s["nf"] = float(s["x"][:, :, 0].float().sum())
        s["loss"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        s["gy"] = torch.empty((B, n ** 3, 16), dtype=torch.bfloat16, device="cuda")
    else:
        g = _gen(seed)
        B, V, K, N = case["B"], case["D"] * case["H"] * case["W"], case["cin"], case["cout"]

        def normal(*shape):
            return torch.randn(shape, generator=g, device="cuda")
        s["x"] = normal(B, V, K).relu().to(torch.bfloat16)
        w = normal(27, K, N) / math.sqrt(27 * K / 2)
        s["wb"] = w.to(torch.bfloat16)                                       # [27][cin][cout]
        s["wf"] = s["wb"].transpose(1, 2).contiguous()                       # [27][cout][cin]
        s["b"] = 0.1 * normal(N)
        s["dy"] = (normal(B, V, N) * (torch.rand((B, V, N), generator=g, device="cuda") < 0.5)).to(torch.bfloat16)
    torch.cuda.synchronize()
    return s


def _train_batch(n, B, g):
    """A batch of media as network input (BF16 [B][V][16]) and targets (FP32 [B][V][4]) of the
    normalised size that the solved flows have."""
    xs, ts = [], []
    for _ in range(B):
        fluid = (_spheres(n, n, n, 6, 0.45, g) == 0).reshape(-1)
        x = torch.zeros((n ** 3, 16), device="cuda")
        x[:, 0] = fluid
        x[:, 1] = fluid
        xs.append(x)
        ts.append(torch.randn((n ** 3, 4), generator=g, device="cuda") * fluid[:, None])
    return torch.stack(xs).to(torch.bfloat16), torch.stack(ts)


# ------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------
_DIR = {"x": 0, "y": 1, "z": 2}


def run(s):
    from paper_1303_2470_gb300 import mp
    case, kind = s["case"], s["kind"]
    if kind in ("slit", "flux"):
        dirs = ("x" if case["flow"] else "z") if kind == "slit" else case["directions"]
        ctx = mp.mp_init_batch(s["solid"], s["u"], s["Db"], s["ka"], s["kd"], directions=dirs,
                               precision="fp64" if kind == "slit" else case["precision"],
                               capacity=case["steps"] + 2, stream=s["stream"])
        for done in range(0, case["steps"], 1024):
            mp.mp_step(ctx, min(1024, case["steps"] - done))
        out = {"series": [mp.mp_vacf(ctx, k, _DIR[d]) for k in range(case["species"]) for d in dirs],
               "density": list(mp.mp_get_field(ctx, 0, 0))}
        ctx.close()
        return out
    if kind == "direct":
        ctx = s["ctx"]
        mp.mp_step(ctx, case["steps"])
        out = {"series": [mp.mp_vacf(ctx, k, _DIR[d]) for k in range(case["species"]) for d in case["directions"]]}
        if case["species"] == 1:
            out["density"] = list(mp.mp_get_field(ctx, 0, 0))  # a checkpoint
        return out
    if kind == "group":
        mp.mp_group_step(s["group"], case["steps"])
        return {"series": [mp.mp_vacf(c, k, 0) for c in s["ctxs"] for k in range(min(10, case["species"]))]}
    if kind == "lb":
        steps, _, _ = mp.lb_steady(s["solid"], (case["force"], 0.0, 0.0), s["u"], tol=1e-7, max_steps=100_000, check_every=100,
                                   rho_out=s["rho"])
        return {"u": s["u"], "rho": s["rho"], "steps": steps}
    if kind == "noalloc":
        mp.mp_step_noalloc(s["solid"], s["u"], 0.05, 5e-3, 5e-3, case["direction"], s["X"], s["Xa"], s["Xn"], s["Xan"],
                           s["Z"])
        return {"X": s["Xn"], "Xa": s["Xan"], "Z": s["Z"]}
    if kind == "warm":
        from paper_1303_2470_gb300 import surrogate
        u, rho = surrogate.warm_start(s["solid"], s["force"], s["model"])
        return {"u": u, "rho": rho}
    if kind == "train":
        m, n, B = s["model"], case["n"], case["batch"]
        y, acts = m.forward(s["x"], B, (n, n, n), keep=True)
        s["loss"].zero_()
        mp.sg_mse(y, 16, s["t"], 4, s["x"], s["gy"], s["loss"], B, n ** 3, s["nf"])
        m.zero_grad()
        m.backward(acts, s["gy"], B, (n, n, n))
        return {"y": y, "loss": s["loss"], "gW": [p["gW"] for p in m.p.values()], "gb": [p["gb"] for p in m.p.values()]}
    B, D, H, W, K, N = (case[k] for k in ("B", "D", "H", "W", "cin", "cout"))
    V = D * H * W
    y = torch.empty((B, V, N), dtype=torch.bfloat16, device="cuda")
    gx = torch.empty((B, V, K), dtype=torch.bfloat16, device="cuda")
    gw = torch.zeros((27, K, N), dtype=torch.float32, device="cuda")
    gb = torch.zeros(N, dtype=torch.float32, device="cuda")
    mp.sg_conv3d(s["x"], s["wf"], s["b"], y, None, B, D, H, W, K, N, 1, True)
    mp.sg_conv3d_wgrad(s["x"], s["dy"], gw, gb, B, D, H, W, K, N)
    mp.sg_conv3d(s["dy"], s["wb"], None, gx, None, B, D, H, W, N, K, -1, False)
    return {"y": y, "gx": gx, "gW": gw, "gb": gb}


# ------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------
_LAYERS = [(0, 16, 32), (0, 32, 32), (1, 32, 64), (1, 64, 64), (2, 64, 96), (2, 96, 96), (3, 96, 128), (3, 128, 128),
           (2, 128, 96), (2, 96, 96), (1, 96, 64), (1, 64, 64), (0, 64, 32), (0, 32, 32), (0, 32, 16)]


def _net_flops(voxels):
    return sum(2.0 * 27 * ci * co * voxels / 8 ** lvl for lvl, ci, co in _LAYERS)


def work(case):
    kind = case["kind"]
    if kind in ("slit", "flux", "direct", "group"):
        if kind == "slit":
            sizes, S, M, eb, por, face = [case["width"] ** 2 * (case["L"] + 2)], case["species"], 1, 8, 1.0, 0.02
        elif kind == "group":
            sizes, S, M, eb, por, face = [case["n%d" % k] ** 3 for k in range(3)], case["species"], 1, 4, 0.4, 0.3
        else:
            fcc = case.get("medium") == "fcc"
            sizes, S, M = [case["nx"] * case["ny"] * case["nz"]], case["species"], len(case["directions"])
            eb, por, face = (2 if case.get("precision") == "fp16" else 4), (0.26 if fcc else 0.4), 0.3
        # per fluid node and species every field read and written once (adsorbed partners on
        # the interface too), the flow (12 B) and node flags (1 B) once per node
        node = S * (1 + M) * 2 * eb * (1.0 + face) + 13
        upd = sum(sizes) * por * case["steps"]
        return {"bytes": upd * node, "flops": upd * S * 18 * (2 * (1 + M) + 2)}
    N = case.get("nx", 0) * case.get("ny", 0) * case.get("nz", 0)
    if kind == "lb":
        # 19 populations read and written per fluid node; the steps to 1e-7 grow with the box
        # and the logarithm of the force (300 at 64^3 and 1e-5, 2400 at 192^3 and 1.8e-3)
        steps = 100 * max(2, round(0.018 * N ** (1 / 3) * math.log(case["force"] / 1e-6)))
        return {"bytes": N * case["porosity"] * 152.0 * steps, "flops": N * case["porosity"] * 300.0 * steps}
    if kind == "noalloc":
        return {"bytes": N * (1 + 4 * 4 + 12.0), "flops": N * 0.4 * 18 * 20}
    if kind == "warm":
        return {"bytes": N * (1 + 16.0), "flops": _net_flops(N)}
    if kind == "train":
        v = case["batch"] * case["n"] ** 3
        # forward, input gradient and weight gradient
        return {"bytes": v * (32 + 16 + 64.0) + 27 * 4 * sum(ci * co for _, ci, co in _LAYERS), "flops": 3 * _net_flops(v)}
    v, K, C = case["B"] * case["D"] * case["H"] * case["W"], case["cin"], case["cout"]
    return {"bytes": v * 4.0 * (K + C) + 27 * K * C * 8.0, "flops": 3 * 2.0 * 27 * v * K * C}


# ------------------------------------------------------------------------------------
# the same results in 64 bits
# ------------------------------------------------------------------------------------
_C = torch.tensor([(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)
                   if 0 < x * x + y * y + z * z < 3])
_WT = [1 / 18 if int((c * c).sum()) == 1 else 1 / 36 for c in _C]
_OPP = [int((_C == -c).all(1).nonzero()) for c in _C]


def _links(solid):
    """Fluid nodes (lattice index), per link the list index of the source r - c (NF where it
    is solid) and the flag of an interfacial node."""
    solid = torch.as_tensor(solid).cuda() != 0
    nf = int((~solid).sum())
    index = torch.full(solid.shape, nf, dtype=torch.long, device="cuda")
    index[~solid] = torch.arange(nf, device="cuda")
    src = torch.stack([torch.roll(index, (int(c[2]), int(c[1]), int(c[0])), (0, 1, 2))[~solid] for c in _C])
    return (~solid), src, (src == nf).any(0)


def _exact_mp(solid, u, Db, ka, kd, dirs, steps):
    """Series [(Z, D) per species and direction] for t = 0..steps + 1 and the density and
    adsorbed density of species 0, dense."""
    fluid, src, itf = _links(solid)
    nf, S = src.shape[1], len(Db)
    f64 = dict(dtype=torch.float64, device="cuda")
    C, W = _C.to(**f64), torch.tensor(_WT, **f64)
    v = torch.zeros((3, nf), **f64) if u is None else u.double()[:, fluid]
    cu = C @ v
    q = W[:, None] * (3 * cu + 4.5 * cu * cu - 1.5 * (v * v).sum(0))
    Db, ka, kd = (torch.as_tensor(np.asarray(t), **f64) for t in (Db, ka, kd))
    opened = src < nf
    pin = torch.empty((S, 18, nf), **f64)
    out = torch.zeros((S, nf), **f64)
    ustar = torch.zeros((S, len(dirs), nf), **f64)
    z0 = torch.zeros((S, len(dirs)), **f64)
    K = torch.where(ka > 0, ka / kd, torch.zeros_like(ka))
    pi = 1.0 / (nf + K * int(itf.sum()))
    P = torch.zeros((S, 1 + len(dirs), nf + 1), **f64)
    stay0 = torch.zeros((S, nf), **f64)
    for i in range(18):
        # link i flows in from r - c; the reverse link flows out to it
        o = _OPP[i]
        qin = torch.cat([q[i], q.new_zeros(1)])[src[i]]
        pin[:, i] = (qin + W[i] * 6 * Db[:, None]) * opened[i]
        po = (q[o] + W[o] * 6 * Db[:, None]) * opened[i]
        out += po
        stay0 += pin[:, i]
        for m, g in enumerate(dirs):
            ustar[:, m] += po * C[o, g]
            z0[:, m] += pi * (po * C[o, g] ** 2).sum(1)
            P[:, 1 + m, :nf] += pi[:, None] * pin[:, i] * C[i, g]
    I = itf.to(torch.float64)
    stay = 1 - out - ka[:, None] * I
    A = torch.zeros((S, 1 + len(dirs), nf), **f64)
    A[:, 0] = (K * pi)[:, None] * I
    P[:, 0, :nf] = pi[:, None] * (stay0 + stay) + kd[:, None] * A[:, 0]
    A[:, 0] = (ka * pi)[:, None] * I + (1 - kd)[:, None] * A[:, 0]
    Z = [z0, (P[:, 1:, :nf] * ustar).sum(2)]
    pa, pd = (ka[:, None] * I)[:, None], kd[:, None, None]
    idx = torch.where(opened, src, torch.full_like(src, nf))
    for _ in range(steps):
        Pn = torch.zeros_like(P)
        acc = P[:, :, :nf] * stay[:, None]
        for i in range(18):
            acc.addcmul_(P.index_select(2, idx[i]), pin[:, i].unsqueeze(1))
        acc += pd * A
        A = pa * P[:, :, :nf] + (1 - pd) * A
        Pn[:, :, :nf] = acc
        P = Pn
        Z.append((P[:, 1:, :nf] * ustar).sum(2))
    Z = torch.stack(Z)                                        # [t][species][direction]
    D = torch.cumsum(Z, 0) - Z[0] / 2
    series = [(Z[:, k, m].cpu().numpy(), D[:, k, m].cpu().numpy()) for k in range(S) for m in range(len(dirs))]

    def dense(a):
        d = torch.zeros(fluid.shape, **f64)
        d[fluid] = a
        return d.cpu().numpy()
    return series, [dense(P[0, 0, :nf]), dense(A[0, 0])]


def _cluster(fluid, src):
    """Fluid-list flags of the largest connected cluster (ties: the one with the smallest node)."""
    nf = src.shape[1]
    lab = torch.arange(nf + 1, device="cuda")
    while True:
        new = torch.minimum(lab[:nf], torch.where(src < nf, lab[src], nf).min(0).values)
        new = torch.minimum(new, new[new])
        if bool((new == lab[:nf]).all()):
            break
        lab = torch.cat([new, lab[nf:]])
    count = torch.bincount(lab[:nf], minlength=nf)
    return lab[:nf] == int((count == count.max()).nonzero()[0])


def _exact_lb(solid, F, tol=1e-7, check=100):
    fluid, src, _ = _links(solid)
    nf = src.shape[1]
    f64 = dict(dtype=torch.float64, device="cuda")
    C = torch.cat([torch.zeros(1, 3), _C.float()]).to(**f64)
    W = torch.tensor([1 / 3] + _WT, **f64)[:, None]
    opp = torch.tensor([0] + [o + 1 for o in _OPP], device="cuda")
    k = torch.arange(nf, device="cuda")
    at = torch.cat([k[None], torch.where(src < nf, src + (torch.arange(1, 19, device="cuda") * nf)[:, None],
                                         (opp[1:] * nf)[:, None] + k)])
    force = torch.tensor(F, **f64)[:, None] * _cluster(fluid, src).to(torch.float64)
    cF = C @ force
    f = torch.zeros((19, nf), **f64)                         # deviations f - w, tau = 1
    prev = torch.zeros((3, nf), **f64)
    t = 0
    while t < 100_000:
        old, f = f, f.reshape(-1)[at]
        drho = f.sum(0)
        u = (C.T @ f + 0.5 * force) / (1 + drho)
        cu = C @ u
        f = W * (drho + (1 + drho) * (3 * cu + 4.5 * cu * cu - 1.5 * (u * u).sum(0)))
        f += 0.5 * W * (3 * cF * (1 + 3 * cu) - 3 * (u * force).sum(0))
        t += 1
        if t % check == 0:
            if float((u - prev).abs().max()) < tol:
                break
            f = 0.5 * (f + old)
        prev = u
    du, dr = torch.zeros((3,) + tuple(fluid.shape), **f64), torch.zeros(tuple(fluid.shape), **f64)
    du[:, fluid] = u
    dr[fluid] = 1 + drho
    return {"u": du, "rho": dr, "steps": None}


def _exact_conv(x, w, b, sign):
    """x [B][D][H][W][K], w [27][K][N] -> [B][D][H][W][N], periodic."""
    y = None
    for t in range(27):
        d = [sign * (t // 9 - 1), sign * (t // 3 % 3 - 1), sign * (t % 3 - 1)]
        p = torch.roll(x, [-v for v in d], (1, 2, 3)) @ w[t]
        y = p if y is None else y.add_(p)
    return y if b is None else y + b


def _exact_net(model, x, B, dims):
    def pool(v):
        s = v.shape
        return v.view(B, s[1] // 2, 2, s[2] // 2, 2, s[3] // 2, 2, s[4]).mean((2, 4, 6))

    def up(v):
        return v.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)

    def conv(name, v):
        p = model.p[name]
        y = _exact_conv(v, p["W"].double(), p["b"].double(), 1)
        return y if name == "out" else y.relu_()
    v = x.double().view((B,) + tuple(dims) + (16,))
    s0 = conv("e0b", conv("e0a", v))
    s1 = conv("e1b", conv("e1a", pool(s0)))
    s2 = conv("e2b", conv("e2a", pool(s1)))
    v = conv("b1", conv("b0", pool(s2)))
    v = conv("d2b", conv("d2a", up(v)) + s2)
    v = conv("d1b", conv("d1a", up(v)) + s1)
    v = conv("d0b", conv("d0a", up(v)) + s0)
    return conv("out", v)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("slit", "flux", "direct"):
        solid, u, Db, ka, kd = _mp_inputs(case, seed)
        dirs = ("x" if case["flow"] else "z") if kind == "slit" else case["directions"]
        series, dens = _exact_mp(solid, u, Db, ka, kd, [_DIR[d] for d in dirs], case["steps"])
        return {"series": series} if kind == "direct" and case["species"] > 1 else {"series": series, "density": dens}
    if kind == "group":
        out = []
        for k in range(3):
            n = case["n%d" % k]
            inp = _mp_inputs({"kind": "group", "nx": n, "ny": n, "nz": n, "species": case["species"]}, seed * 3 + k)
            out += _exact_mp(*inp, [0], case["steps"])[0][:10]
        return {"series": out}
    if kind == "lb":
        g = _gen(seed)
        return _exact_lb(_spheres(case["nx"], case["ny"], case["nz"], case["radius"], case["porosity"], g),
                         (case["force"], 0.0, 0.0))
    s = prepare(case, seed)
    if kind == "noalloc":
        fluid, src, itf = _links(s["solid"])
        nf = src.shape[1]
        C, W = _C.double().cuda(), torch.tensor(_WT, dtype=torch.float64, device="cuda")[:, None]
        v, X, Xa = s["u"].double()[:, fluid], s["X"].double()[fluid], s["Xa"].double()[fluid] * itf
        cu = C @ v
        p = W * (0.3 + 3 * cu + 4.5 * cu * cu - 1.5 * (v * v).sum(0))
        Xn, us = X.clone(), torch.zeros_like(X)
        pX = torch.cat([p * X, p.new_zeros(18, 1)], 1)
        for i in range(18):
            o, opened = _OPP[i], src[i] < nf
            Xn += pX[i][src[i]] - p[o] * X * opened
            if case["direction"] >= 0:
                us += p[o] * C[o, case["direction"]] * opened
        js = (5e-3 * X - 5e-3 * Xa) * itf
        Xn -= js
        dense = [torch.zeros(s["X"].shape, dtype=torch.float64, device="cuda") for _ in range(2)]
        dense[0][fluid], dense[1][fluid] = Xn, (Xa + js) * itf
        z = (Xn * us).sum() if case["direction"] >= 0 else Xn.sum()
        return {"X": dense[0], "Xa": dense[1], "Z": z.reshape(1)}
    if kind == "warm":
        solid = torch.as_tensor(s["solid"]).cuda()
        fluid, src, _ = _links(solid)
        big = torch.zeros(fluid.shape, dtype=torch.bool, device="cuda")
        big[fluid] = _cluster(fluid, src)
        # the network reads the box with the forced axis first (fastest)
        perm = [(0, 1, 2), (0, 2, 1), (1, 2, 0)][case["axis"]]
        comp = [(0, 1, 2), (1, 0, 2), (2, 0, 1)][case["axis"]]
        x = torch.zeros(tuple(fluid.permute(perm).shape) + (16,), dtype=torch.float64, device="cuda")
        x[..., 0], x[..., 1] = fluid.permute(perm), big.permute(perm)
        y = _exact_net(s["model"], x[None], 1, x.shape[:3])[0]
        back = [perm.index(a) for a in range(3)]
        u = torch.zeros((3,) + tuple(fluid.shape), dtype=torch.float64, device="cuda")
        for c in range(3):
            u[comp[c]] = s["force"][case["axis"]] * s["model"].s_u * y[..., c].permute(back) * big
        r = y[..., 3].permute(back)
        rho = 1 + s["force"][case["axis"]] * s["model"].s_rho * (r - r[big].mean()) * big
        return {"u": u, "rho": rho}
    if kind == "train":
        # the gradients pass through BF16 activations in every layer: no 64-bit value of them
        n, B = case["n"], case["batch"]
        y = _exact_net(s["model"], s["x"], B, (n, n, n)).reshape(B, n ** 3, 16)
        m = s["x"][:, :, :1].double()
        loss = ((y[:, :, :4] - s["t"].double()) ** 2 * m).sum() / (4 * s["nf"])
        return {"y": y, "loss": loss.reshape(1), "gW": None, "gb": None}
    B, D, H, W, K, N = (case[k] for k in ("B", "D", "H", "W", "cin", "cout"))
    x, dy = s["x"].double().view(B, D, H, W, K), s["dy"].double().view(B, D, H, W, N)
    wb = s["wb"].double()
    y = _exact_conv(x, wb, s["b"].double(), 1).relu()
    gx = _exact_conv(dy, wb.transpose(1, 2), None, -1)
    gw = torch.stack([torch.roll(x, [-(t // 9 - 1), -(t // 3 % 3 - 1), -(t % 3 - 1)], (1, 2, 3)).reshape(-1, K).T
                      @ dy.reshape(-1, N) for t in range(27)])
    return {"y": y.reshape(B, -1, N), "gx": gx.reshape(B, -1, K), "gW": gw, "gb": dy.reshape(-1, N).sum(0)}
