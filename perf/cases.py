"""What a user of this framework has it do, as cases that can be timed and compared.

Each case is one call pattern through the public entry points (Solver, Ensemble, WarmStartNet) at
a size taken from the workloads, the benchmark or the tests of this repository.  exact() is the
same update in plain torch, FP64, dense arrays and pull streaming, without the package's code.

Solver fields come back as device arrays (Solver.fields_device), cast to the precision the solver
holds them in: FP64, FP32 (as the targets of the warm-start training are), or the 16-bit type that
stores the populations they are sums of (densities, which are 1 plus small deviations, in FP32).
"""
from __future__ import annotations

import math

import numpy as np
import torch

ELEM = {"fp64": (8, 8), "fp32": (4, 4), "fp16": (2, 2), "bf16": (2, 2), "fp16s32": (2, 4), "bf16s32": (2, 4)}
NET_WIDTH = (16, 32, 64, 160)


def listed():
    return [
        # the benchmark's workload: reactive dissolution of a sphere packing, 20 steps and a field read
        {"name": "dissolve256_fp32", "kind": "dissolve", "nx": 256, "ny": 256, "nz": 256, "precision": "fp32", "steps": 20},
        # the same physics on an uneven domain in the accurate 16-bit storage mode
        {"name": "dissolve_uneven_fp16s32", "kind": "dissolve", "nx": 232, "ny": 203, "nz": 181,
         "precision": "fp16s32", "steps": 20},
        # one residual check of the run to steady state that makes and judges warm-start samples:
        # 100 steps at 128^3 with frozen geometry, then the monitors
        {"name": "steady128_fp32", "kind": "steady", "nx": 128, "ny": 128, "nz": 128, "precision": "fp32", "steps": 100},
        # the parity crop of the 3D workload in FP64
        {"name": "crop64_fp64", "kind": "dissolve", "nx": 64, "ny": 64, "nz": 64, "precision": "fp64", "steps": 10},
        # two-component Shan-Chen droplet, the benchmark's second workload
        {"name": "droplet128_fp32", "kind": "droplet", "nx": 128, "ny": 128, "nz": 128, "precision": "fp32", "steps": 10},
        # contact-angle run: a sessile droplet in 2D, walls and adhesion, very many short steps
        {"name": "sessile200x80_fp32", "kind": "sessile", "nx": 200, "ny": 80, "nz": 1, "precision": "fp32", "steps": 100},
        # the smallest workload: the 2D reactive channel in FP64
        {"name": "channel128x64_fp64", "kind": "channel", "nx": 128, "ny": 64, "nz": 1, "precision": "fp64", "steps": 100},
        # the paper's burning channel: velocity inlet, O2, temperature, CO2, conduction in the solid
        {"name": "combustion420x80_fp32", "kind": "combustion", "nx": 420, "ny": 80, "nz": 1, "precision": "fp32",
         "steps": 50},
        # sweep of uneven 2D geometries run to steady state, one residual interval
        {"name": "ensemble2d_fp16", "kind": "ens2d", "members": 12, "lo": 64, "hi": 512, "precision": "fp16", "steps": 50},
        # sweep of uneven 3D geometries
        {"name": "ensemble3d_fp16", "kind": "ens3d", "members": 6, "lo": 64, "hi": 160, "precision": "fp16", "steps": 10},
        # one training step of the warm-start network on a 128^3 sample
        {"name": "net_train128", "kind": "net_train", "nx": 128, "ny": 128, "nz": 128},
        # one prediction of the warm-start network on a smaller uneven domain
        {"name": "net_infer96", "kind": "net_infer", "nx": 128, "ny": 64, "nz": 96},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dissolve", "dissolve", "steady", "droplet", "sessile", "channel", "combustion", "ens2d", "ens3d",
                       "net_train", "net_infer"])
    c = {"kind": kind}
    if kind in ("dissolve", "steady"):
        c["precision"] = rng.choice(["fp32", "fp32", "fp16s32", "bf16s32", "fp16", "bf16", "fp64"])
        hi = 96 if c["precision"] == "fp64" else (256 if kind == "dissolve" else 160)
        for a in ("nx", "ny", "nz"):
            c[a] = _log_int(rng, 40, hi)
        c["steps"] = 20 if kind == "dissolve" else 100
    elif kind == "droplet":
        c["precision"] = rng.choice(["fp32", "fp32", "fp64"])
        for a in ("nx", "ny", "nz"):
            c[a] = _log_int(rng, 32, 128 if c["precision"] == "fp32" else 72)
        c["steps"] = 10
    elif kind == "sessile":
        c.update(nx=_log_int(rng, 120, 600), ny=_log_int(rng, 60, 300), nz=1, precision=rng.choice(["fp32", "fp64"]), steps=50)
    elif kind == "channel":
        c.update(nx=_log_int(rng, 64, 512), ny=_log_int(rng, 32, 256), nz=1, precision=rng.choice(["fp64", "fp32"]), steps=50)
    elif kind == "combustion":
        c.update(nx=_log_int(rng, 100, 840), ny=_log_int(rng, 40, 160), nz=1, precision=rng.choice(["fp32", "fp64"]), steps=20)
    elif kind == "ens2d":
        c.update(members=rng.randint(3, 16), lo=64, hi=_log_int(rng, 128, 512), precision=rng.choice(["fp16", "fp32"]),
                 steps=rng.choice([20, 50]))
    elif kind == "ens3d":
        c.update(members=rng.randint(2, 8), lo=_log_int(rng, 40, 64), hi=_log_int(rng, 80, 160),
                 precision=rng.choice(["fp16", "fp16s32", "fp32"]), steps=10)
    else:
        # multiples of 8 whose coarsest level has a multiple of 128 voxels (the GEMM's tiles)
        while True:
            n = [8 * rng.randint(4, 16) for _ in range(3)]
            if (n[0] // 8) * (n[1] // 8) * (n[2] // 8) % 128 == 0:
                break
        c.update(nx=n[0], ny=n[1], nz=n[2])
    return c


# ------------------------------------------------------------------ inputs

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _spheres(shape, porosity, seed, r_lo=6.0, r_hi=12.0, flag=2):
    """Seeded overlapping spheres (2D: discs) with periodic wrap; their number makes the expected
    porosity the given one.  uint8 flags [nz, ny, nx] on the device."""
    nz, ny, nx = shape
    rng = np.random.default_rng(seed)
    d2 = nz == 1
    p = 2 if d2 else 3
    mean = (r_hi ** (p + 1) - r_lo ** (p + 1)) / ((p + 1) * (r_hi - r_lo)) * (math.pi if d2 else 4.0 / 3.0 * math.pi)
    n = max(1, int(round(-math.log(porosity) * nz * ny * nx / mean)))
    dev = _device()
    c = torch.from_numpy(rng.uniform(0, 1, (n, 3)) * np.array([nz, ny, nx])).to(dev)
    r = torch.from_numpy(rng.uniform(r_lo, r_hi, n)).to(dev)
    if d2:
        c[:, 0] = 0.5
    R = int(math.ceil(r_hi))
    o = torch.arange(-R, R + 1, device=dev)
    oz, oy, ox = torch.meshgrid(torch.zeros(1, dtype=o.dtype, device=dev) if d2 else o, o, o, indexing="ij")
    off = torch.stack([oz.reshape(-1), oy.reshape(-1), ox.reshape(-1)], 1)
    out = torch.zeros(nz * ny * nx, dtype=torch.uint8, device=dev)
    for k in range(0, n, 256):
        b = c[k:k + 256].floor().long()
        q = b[:, None, :] + off[None]
        d = ((q + 0.5 - c[k:k + 256, None, :]) ** 2).sum(-1)
        hit = d <= (r[k:k + 256, None] ** 2)
        idx = ((q[..., 0] % nz) * ny + q[..., 1] % ny) * nx + q[..., 2] % nx
        out[idx[hit]] = flag
    out[0] = 0   # never all solid
    return out.view(nz, ny, nx)


def _modes(shape, seed, count=4):
    """Smooth seeded field of order one, periodic, [nz, ny, nx] FP64 on the device."""
    rng = np.random.default_rng(seed)
    dev = _device()
    ax = [torch.arange(n, device=dev, dtype=torch.float64) / n for n in shape]
    out = torch.zeros(shape, dtype=torch.float64, device=dev)
    for _ in range(count):
        k = rng.integers(-3, 4, 3)
        ph = rng.uniform(0, 2 * math.pi)
        out += torch.sin(2 * math.pi * (k[0] * ax[0][:, None, None] + k[1] * ax[1][None, :, None]
                                        + k[2] * ax[2][None, None, :]) + ph)
    return out / math.sqrt(count / 2.0) / 2.0


def _flow_fields(shape, seed, n_scal, C0=0.6, C1=0.3, u0=0.0185):
    """Fields of a run under way: a mean flow along x with smooth variations, a smooth concentration."""
    s = 10 * seed + 1
    rho = 1.0 + 1e-3 * _modes(shape, s)[None]
    u = torch.stack([u0 * (1.0 + 0.5 * _modes(shape, s + 1)), 0.5 * u0 * _modes(shape, s + 2), 0.5 * u0 * _modes(shape, s + 3)])
    if shape[0] == 1:
        u[2] = 0.0
    C = torch.stack([C0 + C1 * _modes(shape, s + 4 + k) for k in range(n_scal)]) if n_scal else None
    return rho, u, C


def _domain(case, seed):
    """(cfg, flags, (rho, u, C)) of one domain; the arrays are device tensors."""
    kind = case["kind"]
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    shape = (nz, ny, nx)
    prec = case["precision"]
    if kind in ("dissolve", "steady"):
        cfg = dict(dim=3, n_comp=1, tau=[1.0], g=[2.2e-4, 0.0, 0.0], collision="mrt", forcing="guo", n_scal=1,
                   tau_c=[0.5667], J0=0.25, k_react=1.85e-4, ade_open_x=True, C_in=[1.0], periodic=[1, 1, 1],
                   geo_mode="dissolve" if kind == "dissolve" else "none", V_m=1.0, m_s0=1.0, C_ref=[1.0], N_mon=100)
        flags = _spheres(shape, 0.4, seed)
        fields = _flow_fields(shape, seed, 1)
    elif kind == "droplet":
        cfg = dict(dim=3, n_comp=2, tau=[1.0, 1.0], G=[[0.0, 2.7], [2.7, 0.0]], psi_kind="identity", collision="bgk",
                   forcing="guo", n_scal=0, periodic=[1, 1, 1], geo_mode="none")
        flags = torch.zeros(shape, dtype=torch.uint8, device=_device())
        rng = np.random.default_rng(seed)
        a = [torch.arange(n, device=_device(), dtype=torch.float64) - n / 2.0 - rng.uniform(-2, 2) for n in shape]
        r = torch.sqrt(a[0][:, None, None] ** 2 + a[1][None, :, None] ** 2 + a[2][None, None, :] ** 2)
        inside = r < min(shape) / 8.0 * rng.uniform(0.9, 1.1)
        rho = torch.stack([torch.where(inside, 1.0, 0.05), torch.where(inside, 0.05, 1.0)]).to(torch.float64)
        rho *= 1.0 + 1e-3 * _modes(shape, seed)[None]
        fields = (rho, _flow_fields(shape, seed, 0, u0=0.03)[1], None)
    elif kind == "sessile":
        rng = np.random.default_rng(seed)
        g = float(rng.uniform(0.05, 0.15))
        cfg = dict(dim=2, n_comp=2, tau=[1.0, 1.0], G=[[0.0, 2.7], [2.7, 0.0]], psi_kind="identity",
                   G_ads=[g, -g], periodic=[1, 0, 1], rho_solid=0.0, collision="bgk", forcing="guo", n_scal=0)
        flags = torch.zeros(shape, dtype=torch.uint8, device=_device())
        y = torch.arange(ny, device=_device(), dtype=torch.float64)[:, None] + 0.5
        x = torch.arange(nx, device=_device(), dtype=torch.float64)[None, :] - nx / 2.0
        inside = (x * x + y * y < (0.375 * ny) ** 2)[None]
        rho = torch.stack([torch.where(inside, 1.0, 0.05), torch.where(inside, 0.05, 1.0)]).to(torch.float64)
        fields = (rho, _flow_fields(shape, seed, 0, u0=0.03)[1], None)
    elif kind == "channel":
        cfg = dict(dim=2, n_comp=1, tau=[0.8], g=[1e-6, 0.0, 0.0], collision="bgk", forcing="guo", n_scal=1, tau_c=[0.7],
                   J0=0.4, k_react=1e-3, ade_open_x=True, C_in=[1.0], periodic=[1, 1, 1], geo_mode="none")
        flags = _spheres(shape, 0.8, seed, 4.0, 8.0)
        fields = _flow_fields(shape, seed, 1, u0=1e-3)
    elif kind == "combustion":
        r = max(2, ny // 8)
        flags = torch.zeros(shape, dtype=torch.uint8, device=_device())
        y = torch.arange(ny, device=_device(), dtype=torch.float64)[:, None]
        x = torch.arange(nx, device=_device(), dtype=torch.float64)[None, :]
        for k in range(4):
            cx = nx * (0.2 + 0.6 * (k + 0.5) / 4)
            flags[0][(x - cx) ** 2 + (y - (ny - 1) / 2.0) ** 2 <= r * r] = 2
        D = 0.3 * 0.3
        U, k_in, Ta = 1e-2 * D / (2 * r), 3.525e-2 * D / (2 * r), 8.0
        cfg = dict(dim=2, n_comp=1, tau=[0.8], g=[0.0, 0.0, 0.0], collision="bgk", forcing="guo", flow_open_x=True, u_in=U,
                   periodic=[0, 0, 1], n_scal=2, tau_c=[0.8, 0.9], J0=0.4, ade_open_x=True, C_in=[0.22, 1.0],
                   arrhenius=True, arr_A=k_in * math.exp(Ta), arr_Ta=Ta, heat_release=2.0, n_it=24, conjugate=True,
                   tau_s=0.7, c_fs=0.5, product=True, tau_p=0.75, C_in_p=0.0, geo_mode="none")
        rho, u, _ = _flow_fields(shape, seed, 0, u0=U)
        C = torch.stack([0.15 + 0.05 * _modes(shape, seed + 5), 1.1 + 0.1 * _modes(shape, seed + 6),
                         0.05 + 0.02 * _modes(shape, seed + 7)])
        fields = (rho, u, C)
    else:
        raise ValueError(kind)
    return dict(cfg, nx=nx, ny=ny, nz=nz, precision=prec), flags, fields


def _member_sizes(case):
    """Sides of the ensemble's members, spread evenly in the logarithm (fixed by the case, uneven)."""
    n, lo, hi = case["members"], case["lo"], case["hi"]
    return [max(8, int(round(lo * (hi / lo) ** (k / max(1, n - 1)))) + (k % 3) - 1) for k in range(n)]


def _members(case, seed):
    """(cfg, flags, fields) of every member: the reactive channel's transport in 2D, the dissolution's
    in 3D, porosity 0.35 to 0.7."""
    out = []
    for k, s in enumerate(_member_sizes(case)):
        phi = 0.35 + 0.35 * ((k * 0.618) % 1.0)
        sd = 100 * seed + k
        if case["kind"] == "ens2d":
            shape = (1, s, s)
            cfg = dict(dim=2, tau=[0.8], g=[1e-5, 0.0, 0.0], collision="bgk", tau_c=[0.7], J0=0.4, k_react=1e-3, nz=1)
            flags = _spheres(shape, phi, sd, 4.0, 8.0)
            fields = _flow_fields(shape, sd, 1, u0=1e-3)
        else:
            shape = (s, s, s)
            cfg = dict(dim=3, tau=[1.0], g=[2.2e-4, 0.0, 0.0], collision="mrt", tau_c=[0.5667], J0=0.25, k_react=1.85e-4, nz=s)
            flags = _spheres(shape, phi, sd)
            fields = _flow_fields(shape, sd, 1)
        cfg.update(nx=s, ny=s, n_comp=1, forcing="guo", n_scal=1, ade_open_x=True, C_in=[1.0], periodic=[1, 1, 1],
                   geo_mode="none", C_ref=[1.0], precision=case["precision"],
                   N_mon=case["steps"] if case["kind"] == "ens2d" else 0)
        out.append((cfg, flags, fields))
    return out


def _net_plan():
    plan, c = [], 5
    for k, wd in enumerate(NET_WIDTH[:-1]):
        plan += [(f"enc{k}a", c, wd, k), (f"enc{k}b", wd, wd, k)]
        c = wd
    L = len(NET_WIDTH) - 1
    plan += [("mid_a", c, NET_WIDTH[-1], L), ("mid_b", NET_WIDTH[-1], NET_WIDTH[-1], L)]
    c = NET_WIDTH[-1]
    for k in reversed(range(L)):
        plan.append((f"dec{k}", c + NET_WIDTH[k], NET_WIDTH[k], k))
        c = NET_WIDTH[k]
    return plan


def _net_params(seed):
    """He-initialised weights, small biases, as numpy FP32 (insertion order = the network's)."""
    rng = np.random.default_rng(seed)
    p = {}
    for name, ci, co, _ in _net_plan():
        p[name + ".w"] = (rng.standard_normal((co, ci, 3, 3, 3)) * math.sqrt(2.0 / (27 * ci))).astype(np.float32)
        p[name + ".b"] = (0.01 * rng.standard_normal(co)).astype(np.float32)
    p["head.w"] = (rng.standard_normal((4, NET_WIDTH[0])) * math.sqrt(2.0 / NET_WIDTH[0])).astype(np.float32)
    p["head.b"] = (0.01 * rng.standard_normal(4)).astype(np.float32)
    return p


def _net_sample(case, seed):
    """Features (BF16 [V][5]: solid, x, two transport numbers, pore size), targets (FP32 [V][4]) and
    fluid mask (uint8 [V]) of one packing."""
    shape = (case["nz"], case["ny"], case["nx"])
    flags = _spheres(shape, 0.4, seed)
    fluid = (flags == 0)
    d = torch.zeros(shape, device=flags.device)
    left = fluid.float()[None, None]
    for _ in range(10):   # erosions survived: the distance to the solid, up to 10
        d += left[0, 0]
        left = -torch.nn.functional.max_pool3d(-left, 3, 1, 1)
    rng = np.random.default_rng(seed)
    x = torch.empty(shape + (5,), device=flags.device)
    x[..., 0] = (~fluid).float()
    x[..., 1] = (torch.arange(shape[2], device=flags.device) / (shape[2] - 1.0))[None, None, :]
    x[..., 2] = float(rng.uniform(-0.69, 0.0))
    x[..., 3] = float(rng.uniform(-0.69, 0.69))
    x[..., 4] = d / 9.0
    t = torch.stack([_modes(shape, 10 * seed + k, 6) for k in range(4)], -1).float()
    return (x.reshape(-1, 5).to(torch.bfloat16), t.reshape(-1, 4).contiguous(), fluid.reshape(-1).to(torch.uint8), shape)


# ------------------------------------------------------------------ the cases

def _load(solver, flags, fields):
    rho, u, C = fields
    solver.set_geometry(flags.cpu().numpy())
    solver.set_fields(rho.cpu().numpy(), u.cpu().numpy(), None if C is None else C.cpu().numpy())


def prepare(case, seed):
    from paper_2502_12955_gb300 import lbm, surrogate
    kind = case["kind"]
    if kind.startswith("net"):
        net = surrogate.WarmStartNet(width=NET_WIDTH)
        net.set_params(_net_params(seed))
        x, t, fluid, shape = _net_sample(case, seed)
        return {"kind": kind, "net": net, "x": x, "t": t, "fluid": fluid, "n_fluid": int(fluid.sum()), "shape": shape}
    if kind.startswith("ens"):
        mem = _members(case, seed)
        e = lbm.Ensemble([c for c, _, _ in mem])
        for (_, flags, fields), m in zip(mem, e.members):
            _load(m, flags, fields)
        return {"kind": kind, "e": e, "steps": case["steps"], "dtype": _dtypes(case["precision"])}
    cfg, flags, fields = _domain(case, seed)
    s = lbm.Solver(cfg)
    _load(s, flags, fields)
    return {"kind": kind, "s": s, "steps": case["steps"], "dtype": _dtypes(case["precision"])}


def _dtypes(precision):
    full = torch.float64 if precision == "fp64" else torch.float32
    flow = {"fp16": torch.float16, "bf16": torch.bfloat16}.get(precision[:4], full)
    scal = full if precision.endswith("s32") else flow
    return {"rho": full, "u": flow, "C": scal, "acc": scal, "flags": torch.uint8}


def _fields(s, dtype, keys):
    f = s.fields_device()
    return {k: torch.as_tensor(f[k], device="cuda").to(dtype[k]) for k in keys if k in f}


def run(state):
    kind = state["kind"]
    if kind == "net_infer":
        return state["net"].forward(state["x"], state["shape"])
    if kind == "net_train":
        net = state["net"]
        loss = net.train_step(state["x"], state["t"], state["fluid"], state["n_fluid"], state["shape"], lr=1e-3)
        return {"loss": loss.float(), "grads": net.gflat, "weights": net.flat}
    if kind.startswith("ens"):
        e = state["e"]
        if kind == "ens2d":
            e.run_to_steady(1e-14, state["steps"])
        else:
            e.step(state["steps"])
        return [_fields(m, state["dtype"], ("rho", "u", "C", "acc")) for m in e.members]
    s = state["s"]
    s.step(state["steps"])
    if kind in ("droplet", "sessile"):
        return _fields(s, state["dtype"], ("rho", "u"))
    out = {}
    if kind == "steady":
        m = s.monitors()
        out["monitors"] = {k: torch.tensor(m[k], dtype=state["dtype"]["rho"]) for k in ("mass0", "species0", "reacted", "nfluid", "residual")}
    out.update(_fields(s, state["dtype"], ("rho", "u", "C", "acc", "flags")))
    return out


def work(case):
    """Populations read and written once per fluid node and step, the fields of the read-back once."""
    kind = case["kind"]
    if kind.startswith("net"):
        V = case["nx"] * case["ny"] * case["nz"]
        flops = sum(2.0 * 27 * ci * co * (V >> (3 * k)) for _, ci, co, k in _net_plan()) + 2.0 * 16 * 4 * V
        acts = sum(2.0 * (ci + co) * (V >> (3 * k)) for _, ci, co, k in _net_plan()) + V * (2 * 16 + 16)
        return {"bytes": acts if kind == "net_infer" else 3 * acts + V * 37, "flops": flops if kind == "net_infer" else 3 * flops}
    ef, es = ELEM[case["precision"]]
    d3 = kind in ("dissolve", "steady", "droplet", "ens3d")
    q, qc = (19, 7) if d3 else (9, 5)
    if kind.startswith("ens"):
        n = [s ** 3 if d3 else s * s for s in _member_sizes(case)]
        fluid = sum(v * (0.35 + 0.35 * ((k * 0.618) % 1.0)) for k, v in enumerate(n))
        nodes = sum(n)
    else:
        nodes = case["nx"] * case["ny"] * case["nz"]
        fluid = nodes * {"dissolve": 0.4, "steady": 0.4, "channel": 0.8, "combustion": 0.94}.get(kind, 1.0)
    nc, ns = {"droplet": (2, 0), "sessile": (2, 0), "combustion": (1, 3)}.get(kind, (1, 1))
    out = 4 * (nc + 3 + ns) * (2 if case["precision"] == "fp64" else 1)
    flops = nc * (16.0 * q if not d3 else 14.0 * q) + ns * 5.0 * qc + (110.0 if kind in ("dissolve", "steady", "ens3d") else 0.0)
    return {"bytes": 2.0 * fluid * (ef * q * nc + es * qc * ns) * case["steps"] + nodes * out, "flops": fluid * flops * case["steps"]}


# ------------------------------------------------------------------ the same in 64 bits

def _lattice(dim):
    """Directions and weights of D3Q19 / D2Q9 (the first 7 / 5 are the scalar lattice's)."""
    if dim == 3:
        c = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
        c += [(s * a, s * b, s * d) for (a, b, d) in ((1, 1, 0), (1, 0, 1), (0, 1, 1), (1, -1, 0), (1, 0, -1), (0, 1, -1)) for s in (1, -1)]
        w = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
    else:
        c = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)]
        w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
    return c, w, [c.index((-a, -b, -d)) for a, b, d in c]


def _relaxation(cfg, c):
    """The collision matrix: f* = f - A (f - f_eq + F / 2) + F."""
    om = 1.0 / cfg["tau"][0]
    if cfg["collision"] != "mrt":
        return None
    x, y, z = (np.array([v[a] for v in c], float) for a in range(3))
    c2 = x * x + y * y + z * z
    one = np.ones_like(x)
    rows = [(one, om), (19 * c2 - 30, 1.19), ((21 * c2 * c2 - 53 * c2 + 24) / 2, 1.4), (x, om), ((5 * c2 - 9) * x, 1.2), (y, om),
            ((5 * c2 - 9) * y, 1.2), (z, om), ((5 * c2 - 9) * z, 1.2), (3 * x * x - c2, om), ((3 * c2 - 5) * (3 * x * x - c2), om),
            (y * y - z * z, om), ((3 * c2 - 5) * (y * y - z * z), om), (x * y, om), (y * z, om), (x * z, om),
            (x * (y * y - z * z), 1.98), (y * (z * z - x * x), 1.98), (z * (x * x - y * y), 1.98)]
    M = np.array([r for r, _ in rows])
    return np.linalg.inv(M) @ np.diag([s for _, s in rows]) @ M


class _Reference:
    """The update of one domain on dense FP64 arrays [q, nz, ny, nx]; state = populations at the start of
    a step.  Solid nodes carry zeros."""

    def __init__(self, cfg, flags, fields):
        self.cfg, self.flags = cfg, flags
        dev = flags.device
        self.c, self.w, self.opp = _lattice(cfg["dim"])
        self.qc = 7 if cfg["dim"] == 3 else 5
        J0 = cfg.get("J0", 0.25)
        self.wc = [J0] + [(1 - J0) / (self.qc - 1)] * (self.qc - 1)
        self.ics2 = (self.qc - 1) / (2.0 * (1 - J0))
        self.nc, self.ng = cfg["n_comp"], cfg["n_scal"]
        self.ns = self.ng + int(cfg.get("product", False))
        self.tc = list(cfg.get("tau_c", []))[:self.ng] + ([cfg["tau_p"]] if cfg.get("product") else [])
        self.cin = list(cfg.get("C_in", []))[:self.ng] + ([cfg["C_in_p"]] if cfg.get("product") else [])
        A = _relaxation(cfg, self.c)
        self.A = None if A is None else torch.from_numpy(A).to(dev)
        per = list(cfg["periodic"])
        self.fluid = flags == 0
        fl = self.fluid
        per_c = [per[0] and not cfg.get("ade_open_x"), per[1], per[2]]
        self.src = [self._from(fl, c, per) & fl for c in self.c]              # x - c is a fluid node
        self.src_c = [self._from(fl, c, per_c) & fl for c in self.c[:self.qc]]
        self.react = [self._from(flags == 2, c, per_c) & fl for c in self.c[:self.qc]]
        self.sol = [self._from(~fl, c, per_c) & fl for c in self.c[:self.qc]]
        rho, u, C = fields
        self.f = torch.stack([torch.stack([self._feq(i, rho[s], u) for i in range(len(self.c))]) for s in range(self.nc)]) * fl
        self.h = None
        if self.ns:
            self.h = torch.stack([torch.stack([self.wc[j] * C[s] * (1 + self.ics2 * self._cu(j, u)) for j in range(self.qc)])
                                  for s in range(self.ns)]) * fl
        self.acc = torch.zeros(flags.shape, dtype=torch.float64, device=dev)
        self.conj = bool(cfg.get("conjugate"))
        if self.conj:
            self.g = torch.stack([w * C[1] for w in self.wc]) * ~fl
            self.kb = None

    @staticmethod
    def _from(a, c, per):
        """a at x - c; False / 0 beyond a closed face."""
        out = torch.roll(a, (c[2], c[1], c[0]), (0, 1, 2))
        for axis, s, p in ((2, c[0], per[0]), (1, c[1], per[1]), (0, c[2], per[2])):
            if s and not p:
                out = out.clone()
                out.select(axis, 0 if s > 0 else -1).zero_()
        return out

    def _cu(self, i, u):
        out = 0.0
        for a in range(3):
            if self.c[i][a]:
                out = out + self.c[i][a] * u[a]
        return out

    def _feq(self, i, rho, u):
        cu = self._cu(i, u)
        return self.w[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u * u).sum(0))

    def _closed(self):
        """Scalar populations with the reactive links closed, and the rate k C_b of each link."""
        cfg, h = self.cfg, self.h
        out, rates = h.clone(), {}
        for j in range(1, self.qc):
            if not self.react[j].any():
                continue
            m, hb, w = self.react[j], h[0, self.opp[j]], self.wc[j]
            fc = self.tc[0] / (self.tc[0] - 0.5)
            if self.conj:
                if self.kb is not None:
                    k = self.kb[j]
                else:
                    T = (cfg["c_fs"] * h[1].sum(0) + self._from(self.g.sum(0), self.c[j], [1, 1, 1])) / (cfg["c_fs"] + 1)
                    k = cfg["arr_A"] * torch.exp(-cfg["arr_Ta"] / torch.where(m, T, 1.0))
            else:
                k = cfg["k_react"]
            cb = 2 * hb / (2 * w + k * fc)
            out[0, j] = torch.where(m, 2 * w * cb - hb, h[0, j])
            rates[j] = torch.where(m, k * cb, 0.0)
            if cfg.get("product"):
                fp = self.tc[-1] / (self.tc[-1] - 0.5)
                out[-1, j] = torch.where(m, h[-1, self.opp[j]] + rates[j] * fp, h[-1, j])
        return out, rates

    def _forces(self, rho):
        cfg = self.cfg
        F = [torch.stack([rho[s] * cfg["g"][a] for a in range(3)]) if any(cfg.get("g", [0])) else
             torch.zeros((3,) + rho.shape[1:], dtype=torch.float64, device=rho.device) for s in range(self.nc)]
        if self.nc == 2:   # psi = rho, cross cohesion, adhesion at walls (no solid psi)
            for s in range(2):
                G = cfg["G"][s][1 - s]
                other = rho[1 - s]
                for i in range(1, len(self.c)):
                    back = tuple(-v for v in self.c[i])
                    nb = self._from(other, back, cfg["periodic"])
                    wall = self.fluid & ~self._from(self.fluid, back, cfg["periodic"])
                    for a in range(3):
                        if self.c[i][a]:
                            F[s][a] -= rho[s] * G * self.w[i] * self.c[i][a] * nb
                            if "G_ads" in cfg:
                                F[s][a] -= rho[s] * cfg["G_ads"][s] * self.w[i] * self.c[i][a] * wall
        return F

    def _macros(self):
        rho = self.f.sum(1)
        F = self._forces(rho)
        j = 0.0
        for s in range(self.nc):
            j = j + 0.5 * F[s] + torch.stack([sum(self.c[i][a] * self.f[s, i] for i in range(len(self.c)) if self.c[i][a])
                                              if any(v[a] for v in self.c) else torch.zeros_like(rho[0]) for a in range(3)])
        u = j / torch.where(self.fluid, rho.sum(0), 1.0)
        return rho, F, u * self.fluid

    def step(self):
        cfg = self.cfg
        rho, F, u = self._macros()
        closed, rates = self._closed() if self.ns else (None, {})
        for j, r in rates.items():
            self.acc += torch.roll(r, (-self.c[j][2], -self.c[j][1], -self.c[j][0]), (0, 1, 2))
        new = torch.zeros_like(self.f)
        for s in range(self.nc):
            uF = (u * F[s]).sum(0)
            post = torch.empty_like(self.f[s])
            Fi = torch.stack([self.w[i] * (3 * (self._cu(i, F[s]) - uF) + 9 * self._cu(i, u) * self._cu(i, F[s]))
                              for i in range(len(self.c))])
            n = self.f[s] - torch.stack([self._feq(i, rho[s], u) for i in range(len(self.c))]) + 0.5 * Fi
            n = n / cfg["tau"][s] if self.A is None else (self.A @ n.reshape(len(self.c), -1)).reshape(n.shape)
            post = self.f[s] - n + Fi
            del n, Fi
            for i in range(len(self.c)):
                v = torch.where(self.src[i], self._from(post[i], self.c[i], [1, 1, 1]), post[self.opp[i]])
                if cfg.get("flow_open_x"):
                    ny = cfg["ny"]
                    sy = (torch.arange(ny, dtype=torch.float64, device=v.device) + 0.5) / ny
                    if self.c[i][0] > 0:
                        v[:, :, 0] += 6 * self.w[i] * rho[s][:, :, 0] * (6 * cfg["u_in"] * sy * (1 - sy))[None]
                    elif self.c[i][0] < 0:
                        v[:, :, -1] = post[i][:, :, -1]
                new[s, i] = v * self.fluid
        if self.ns:
            hnew = torch.zeros_like(self.h)
            for s in range(self.ns):
                C = closed[s].sum(0)
                post = torch.stack([closed[s, j] - (closed[s, j] - self.wc[j] * C * (1 + self.ics2 * self._cu(j, u))) / self.tc[s]
                                    for j in range(self.qc)])
                if s == 1 and self.conj:
                    tpost = post
                for j in range(self.qc):
                    v = torch.where(self.src_c[j], self._from(post[j], self.c[j], [1, 1, 1]), post[self.opp[j]])
                    if cfg.get("ade_open_x") and self.c[j][0] > 0:
                        v[:, :, 0] = self.wc[j] * self.cin[s] * (1 + self.ics2 * self._cu(j, u)[:, :, 0])
                    elif cfg.get("ade_open_x") and self.c[j][0] < 0:
                        v[:, :, -1] = post[j][:, :, -1]
                    hnew[s, j] = v * self.fluid
            if self.conj:
                self._conduct(tpost, hnew)
            self.h = hnew
        self.f = new

    def _conduct(self, tpost, hnew):
        """The solid's heat lattice and its exchange with the fluid temperature across every solid link."""
        cfg = self.cfg
        per_c = [cfg["periodic"][0] and not cfg.get("ade_open_x"), cfg["periodic"][1], cfg["periodic"][2]]
        solid = ~self.fluid
        Ts = self.g.sum(0)
        gp = torch.stack([self.g[q] - (self.g[q] - self.wc[q] * Ts) / cfg["tau_s"] for q in range(self.qc)])
        gnew = torch.zeros_like(self.g)
        for q in range(self.qc):
            ok = self._from(solid, self.c[q], per_c) & solid
            gnew[q] = torch.where(ok, self._from(gp[q], self.c[q], [1, 1, 1]), gp[self.opp[q]]) * solid
        fc = self.tc[0] / (self.tc[0] - 0.5)
        cf, w = cfg["c_fs"], self.wc[1]
        kb = {}
        for i in range(1, self.qc):   # arriving at the fluid node in direction i from the solid node x - c_i
            j = self.opp[i]
            m, mr = self.sol[i], self.react[i]
            ho, go = tpost[j], self._from(gp[i], self.c[i], [1, 1, 1])
            T0 = torch.where(m, (cf * ho + go) / (w * (cf + 1)), 1.0)
            T, k = T0, None
            hb = hnew[0, j]
            for _ in range(cfg["n_it"] + 1):
                k = cfg["arr_A"] * torch.exp(-cfg["arr_Ta"] / T)
                Q = cfg["heat_release"] * k * 2 * hb / (2 * w + k * fc)
                T = torch.where(mr, T0 + 0.5 * cf * Q / (w * (cf + 1)), T0)
            kb[i] = k
            hnew[1, i] = torch.where(m, 2 * w * T - ho, hnew[1, i])
            back = torch.where(m, 2 * w * T - go, 0.0)
            hit = torch.roll(m, (-self.c[i][2], -self.c[i][1], -self.c[i][0]), (0, 1, 2))
            gnew[j] = torch.where(hit, torch.roll(back, (-self.c[i][2], -self.c[i][1], -self.c[i][0]), (0, 1, 2)), gnew[j])
        self.g, self.kb = gnew, kb

    def fields(self):
        rho, _, u = self._macros()
        out = {"rho": rho, "u": u}
        if self.ns:
            out["C"] = self._closed()[0].sum(1)
            if self.conj:
                out["C"][1] += self.g.sum(0)
            out["acc"] = self.acc
        return out


def _net_exact(case, seed):
    x, t, fluid, shape = _net_sample(case, seed)
    dev = x.device
    p = {k: torch.from_numpy(v).to(dev, torch.float64) for k, v in _net_params(seed).items()}
    train = case["kind"] == "net_train"
    if train:
        for v in p.values():
            v.requires_grad_(True)
    F = torch.nn.functional
    with torch.set_grad_enabled(train):
        h = x.double().reshape(shape + (5,)).permute(3, 0, 1, 2)[None]
        conv = lambda n, v: F.relu(F.conv3d(v, p[n + ".w"], p[n + ".b"], padding=1))  # noqa: E731
        skips = []
        for k in range(len(NET_WIDTH) - 1):
            h = conv(f"enc{k}b", conv(f"enc{k}a", h))
            skips.append(h)
            h = F.avg_pool3d(h, 2)
        h = conv("mid_b", conv("mid_a", h))
        for k in reversed(range(len(NET_WIDTH) - 1)):
            h = conv(f"dec{k}", torch.cat([F.interpolate(h, scale_factor=2), skips[k]], 1))
        y = torch.einsum("oc,cv->vo", p["head.w"], h[0].reshape(NET_WIDTH[0], -1)) + p["head.b"]
        if not train:
            return y
        loss = (((y - t.double()) * fluid[:, None]) ** 2).sum() / (int(fluid.sum()) * 4)
        loss.backward()
    g = torch.cat([v.grad.reshape(-1) for v in p.values()])
    w = torch.cat([v.detach().reshape(-1) for v in p.values()])
    return {"loss": loss.detach().reshape(1), "grads": g, "weights": w - 1e-3 * g / (g.abs() + 1e-8)}


def exact(case, seed):
    kind = case["kind"]
    if kind.startswith("net"):
        return _net_exact(case, seed)
    out = []
    for cfg, flags, fields in (_members(case, seed) if kind.startswith("ens") else [_domain(case, seed)]):
        r = _Reference(cfg, flags, fields)
        for _ in range(case["steps"]):
            r.step()
        f = r.fields()
        if kind.startswith("ens"):
            out.append(f)
            continue
        if kind == "steady":
            f["monitors"] = {"mass0": r.f.sum(), "species0": r.h[0].sum(), "reacted": r.acc.sum(),
                             "nfluid": r.fluid.sum().double(), "residual": None}
        if "acc" in f:
            f["flags"] = flags   # no node dissolves in the first pass
        return f
    return out
