"""The workloads this solver is timed on, and their inputs, passes and FP64 answers.

A case is a flow problem and a number of time steps.  One pass advances the
flow by that many steps from where the last pass left it, reads the last check
step's residual and flow rate where the case has check steps, and reads the
density and velocity fields back into device memory: what a program that
monitors a transient or a march to steady state does between two of its own
looks at the flow.  Flows start from rest.

Fields are returned in the precision that the populations are stored in.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1610_01388_gb300 import lbm
from paper_1610_01388_gb300 import workloads as W

TORCH_TYPE = {"F64": torch.float64, "F32": torch.float32, "F16": torch.float16,
              "BF16": torch.bfloat16}
# scalars of the bfloat16 form go back as half, numpy's 16-bit float
SCALAR_TYPE = {"F64": np.float64, "F32": np.float32, "F16": np.float16, "BF16": np.float16}
STORED_BYTES = {"F64": 8, "F32": 4, "F16": 2, "BF16": 2}
VELOCITIES = {"D2Q9": 9, "D3Q15": 15, "D3Q19": 19, "D3Q27": 27}
NU = 0.1                # plastic viscosity
M = 1e6                 # Papanastasiou regularisation (1e4 on the plane channel)


def _case(name, kind, lattice, model, storage, nx, ny, nz, steps, check_every=0, layout="dense"):
    c = {"kind": kind, "lattice": lattice, "model": model, "storage": storage, "nx": nx, "ny": ny,
         "nz": nz, "steps": steps, "check_every": check_every, "layout": layout}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the paper's plane Bingham-Poiseuille channel, marched to steady
        # state in double precision: 256 cells, the smallest problem
        _case("channel_4x64_f64_ir", "channel", "D2Q9", "IR", "F64", 4, 64, 1, 2000),
        # the paper's periodic cylinder cell (creeping-flow table), watched
        # through its residual
        _case("cylinder_80_f64_pr", "cylinder", "D2Q9", "PR", "F64", 80, 80, 1, 500, 250),
        # the paper's square duct of 63 lattice units, one cell long, in
        # double precision
        _case("duct_63_f64_ir", "duct", "D3Q27", "IR", "F64", 1, 64, 64, 200),
        # a channel of the serving mix on its own
        _case("channel_128_f32_pr", "channel", "D2Q9", "PR", "F32", 128, 66, 1, 1000),
        # a small porous sample with odd sides, watched through its residual
        _case("porous_45_f32_pr", "porous", "D3Q15", "PR", "F32", 45, 47, 43, 400, 200),
        # the start-up of the square duct, both models: the headline workload
        _case("duct_256_f32_ir", "duct", "D3Q27", "IR", "F32", 256, 128, 128, 100, 50),
        _case("duct_256_f32_pr", "duct", "D3Q27", "PR", "F32", 256, 128, 128, 100, 50),
        # the porous box in the layout made for it, plain and reduced precision
        _case("porous_256_f32_ir", "porous", "D3Q19", "IR", "F32", 256, 256, 256, 100, 50, "compact"),
        _case("porous_256_f16_pr", "porous", "D3Q19", "PR", "F16", 256, 256, 256, 100, 0, "compact"),
        # the precision workload's long duct, the largest problem
        _case("duct_512_f16_pr", "duct", "D3Q27", "PR", "F16", 512, 192, 192, 60),
        # the other 16-bit form
        _case("duct_256_bf16_ir", "duct", "D3Q27", "IR", "BF16", 256, 128, 128, 100),
        # many resident domains of the serving mix stepped together
        {"name": "mix_48", "kind": "mix", "requests": 48, "steps": 200, "check_every": 100},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["channel", "channel", "cylinder", "duct", "duct", "duct", "porous", "porous",
                       "porous", "mix"])
    model = rng.choice(["IR", "PR"])
    if kind == "mix":
        return {"kind": "mix", "requests": rng.randrange(8, 57), "steps": rng.randrange(50, 151),
                "check_every": 50}
    if kind in ("channel", "cylinder"):
        storage = rng.choice(["F64", "F64", "F32", "F16"])
        if kind == "channel":
            nx, ny = rng.choice([4, _log(rng, 4, 128)]), rng.randrange(17, 258)
        else:
            nx = ny = rng.randrange(40, 161)
        steps = min(_log(rng, 100, 2000), 12_000_000 // (nx * ny))
        check = rng.choice([0, max(2, steps // 2)])
        return _case(None, kind, "D2Q9", model, storage, nx, ny, 1, steps, check)
    lattice = rng.choice(["D3Q15", "D3Q19", "D3Q19", "D3Q27", "D3Q27"])
    storage = rng.choice(["F32", "F32", "F32", "F16", "F16", "F64"])
    if kind == "duct" and storage == "F16":
        storage = rng.choice(["F16", "BF16"])    # BF16 does not resolve the porous flows
    top = 40_000 if storage == "F64" else 8_000_000
    if kind == "duct":
        side = _log(rng, 18, 193)
        nx = max(1, min(_log(rng, 1, 512), top // (side * side)))
        dims = (nx, side, side)
    else:
        side = _log(rng, 24, 34 if storage == "F64" else 200)
        dims = (side + rng.randrange(-3, 4), side, side + rng.randrange(-3, 4))
    cells = dims[0] * dims[1] * dims[2]
    # no more than about a quarter of the largest listed case's cell steps
    steps = max(10, min(_log(rng, 20, 1000), 250_000_000 // cells,
                        3_000_000 // cells if storage == "F64" else 1000))
    check = rng.choice([0, steps // 2])
    layout = rng.choice(["dense", "compact"]) if kind == "porous" else "dense"
    return _case(None, kind, lattice, model, storage, *dims, steps, check, layout)


# --- inputs -------------------------------------------------------------------

@functools.lru_cache(maxsize=8)
def _porous(nx, ny, nz):
    small = min(nx, ny, nz) < 96
    return W.porous_mask((nx, ny, nz), porosity=0.7, r_min=3.0 if small else 6.0,
                         r_max=5.0 if small else 10.0, seed=1, max_attempts=400_000)[0]


def _flow(case, seed):
    """Mask and rheology of one domain, from the seed: the Bingham number, the
    force and, in porous boxes, where the periodic box is cut."""
    r = np.random.Generator(np.random.PCG64([seed, 11]))
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["kind"] == "channel":
        p = W.channel_params(H=ny - 1, nu_p=NU, u_newton=float(r.uniform(0.008, 0.015)),
                             bn=float(r.uniform(0.1, 10.0)))
        mask, m = W.channel_mask(nx, ny), 1e4 if nx == 4 else M
    elif case["kind"] == "cylinder":
        g = float(r.uniform(1.0e-6, 1.5e-6))
        p = {"g": g, "sigma_y": g * nx * float(r.uniform(0.01, 0.02))}
        mask, m = W.cylinder_mask(nx, 0.4 * nx), M
    elif case["kind"] == "duct":
        p = W.duct_params(H=ny - 1, nu_p=NU, u_newton=float(r.uniform(0.015, 0.025)),
                          bn=float(r.uniform(0.5, 8.0)))
        mask, m = W.duct_mask(nx, ny, nz), M
    else:
        # a priori Bn on the mean grain diameter, below the nearly jammed flows
        p = W.porous_params(nu_p=NU, d_mean=8.0 if min(nx, ny, nz) < 96 else 16.0,
                            g=float(r.uniform(1.5e-5, 2.5e-5)), bn=float(r.uniform(0.1, 0.5)))
        shift = tuple(int(r.integers(n)) for n in (nz, ny, nx))
        mask, m = np.roll(_porous(nx, ny, nz), shift, axis=(0, 1, 2)), M
    return mask, {"mu_p": NU, "sigma_y": float(p["sigma_y"]), "m": m, "g": (float(p["g"]), 0.0, 0.0)}


def _mix(case, seed):
    """The serving mix: channels, ducts and porous boxes of the scaled stream,
    in FP16 but for the nearly jammed porous boxes, which need FP32.  Which
    domains are resident follows from their number; their forces, yield
    stresses and, in porous boxes, where the box is cut, from the seed."""
    got = W.serving_requests(n=case["requests"], rate=150.0, seed=8, storage="F16",
                             channel_widths=(16, 64), channel_length=128, duct_sides=(16, 48),
                             duct_length=32, porous_sides=(24, 48), porous_radius=(3.0, 5.0),
                             porous_pool=2)
    r = np.random.Generator(np.random.PCG64([seed, 13]))
    for q in got:
        a, b = float(r.uniform(0.8, 1.2)), float(r.uniform(0.8, 1.2))
        q["g"] = tuple(a * x for x in q["g"])
        q["sigma_y"] *= a * b
        shift = tuple(int(r.integers(n)) for n in q["mask"].shape)
        if q["kind"] == "porous":
            q["mask"] = np.roll(q["mask"], shift, axis=(0, 1, 2))
            if q["bn"] >= 1.0:
                q["storage"] = "F32"
    return got


def _params(q):
    return {k: q[k] for k in ("mu_p", "sigma_y", "m", "g")}


def prepare(case, seed):
    if case["kind"] == "mix":
        batch = lbm.Batch(64 << 30, case["check_every"],
                          stream=torch.cuda.current_stream().cuda_stream)
        doms = []
        for q in _mix(case, seed):
            i = batch.add(q["lattice"], q["mask"], model=q["model"], storage=q["storage"], **_params(q))
            doms.append((i, q["storage"], torch.empty(4, q["mask"].size, dtype=torch.float64,
                                                      device="cuda")))
        return {"case": case, "batch": batch, "doms": doms}
    mask, p = _flow(case, seed)
    s = lbm.Solver(case["lattice"], mask, model=case["model"], storage=case["storage"],
                   layout=case["layout"], check_every=case["check_every"], use_torch=True, **p)
    return {"case": case, "solver": s,
            "out": torch.empty(4, mask.size, dtype=torch.float64, device="cuda")}


def _read(handle, out):
    lbm.lbm_fields_device(handle, *(out[k].data_ptr() for k in range(4)))


def run(state):
    case = state["case"]
    if case["kind"] == "mix":
        batch = state["batch"]
        batch.step(case["steps"])
        got = {}
        for i, storage, out in state["doms"]:
            flow = batch.status(i).flow[0]
            _read(batch.solver(i), out)
            g = got.setdefault(storage, {"flow": [], "rho": [], "u": []})
            g["flow"].append(flow)
            g["rho"].append(out[0])
            g["u"].append(out[1:].reshape(-1))
        return {k: {"flow": np.array(g["flow"], SCALAR_TYPE[k]),
                    "rho": torch.cat(g["rho"]).to(TORCH_TYPE[k]),
                    "u": torch.cat(g["u"]).to(TORCH_TYPE[k])} for k, g in got.items()}
    s, out, kind = state["solver"], state["out"], TORCH_TYPE[case["storage"]]
    s.step(case["steps"])
    got = {}
    if case["check_every"]:
        residual, _, flow = s.residual()
        scalar = SCALAR_TYPE[case["storage"]]
        got = {"residual": scalar(residual), "flow": scalar(flow)}
    _read(s.h, out)
    return dict(got, rho=out[0].to(kind), u=out[1:].to(kind))


# --- what a pass cannot do without ------------------------------------------------

def _domain_work(lattice, model, storage, cells, fluid, steps):
    q, b = VELOCITIES[lattice], STORED_BYTES[storage]
    # per fluid cell and step: the populations in and out, the cell's mask
    # byte and, for PR, the relaxation time in and out; then the fields
    tau = 2 * max(b, 4) if model == "PR" else 0
    return {"bytes": steps * fluid * (2 * q * b + 1 + tau) + 32 * cells,
            "flops": steps * fluid * (9 * q + 40)}


def work(case):
    total = {"bytes": 0.0, "flops": 0.0}
    if case["kind"] == "mix":
        parts = [(q["lattice"], q["model"], q["storage"], q["mask"]) for q in _mix(case, 7)]
    else:
        parts = [(case["lattice"], case["model"], case["storage"], _flow(case, 7)[0])]
    for lattice, model, storage, mask in parts:
        w = _domain_work(lattice, model, storage, mask.size, int((mask == 0).sum()), case["steps"])
        total = {k: total[k] + w[k] for k in total}
    return total


# --- the same flow in FP64, by plain tensor arithmetic -----------------------------

def _velocity_set(lattice):
    d = 2 if lattice == "D2Q9" else 3
    keep = {"D2Q9": (0, 1, 2), "D3Q15": (0, 1, 3), "D3Q19": (0, 1, 2), "D3Q27": (0, 1, 2, 3)}[lattice]
    weight = {"D2Q9": (4 / 9, 1 / 9, 1 / 36, 0), "D3Q15": (2 / 9, 1 / 9, 0, 1 / 72),
              "D3Q19": (1 / 3, 1 / 18, 1 / 36, 0), "D3Q27": (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[lattice]
    c = [(x, y, z) for z in ((0,) if d == 2 else (-1, 0, 1)) for y in (-1, 0, 1) for x in (-1, 0, 1)
         if abs(x) + abs(y) + abs(z) in keep]
    return d, c, [weight[sum(map(abs, v))] for v in c]


def _march(lattice, model, mask, steps, check_every, mu_p, sigma_y, m, g, gdot_c=1e-8, magic=0.25):
    """h = f - w from rest through `steps` pull-and-collide steps in FP64."""
    dim, c, w = _velocity_set(lattice)
    Q, dev = len(c), "cuda"
    opp = [c.index((-x, -y, -z)) for x, y, z in c]
    solid = torch.from_numpy(np.ascontiguousarray(mask)).to(dev) != 0
    n = solid.numel()
    cell = torch.arange(n, device=dev).reshape(solid.shape)
    src = torch.empty(Q, n, dtype=torch.int64, device=dev)
    for i, (x, y, z) in enumerate(c):
        from_cell = torch.roll(cell, (z, y, x), (0, 1, 2))
        from_solid = torch.roll(solid, (z, y, x), (0, 1, 2))
        src[i] = torch.where(from_solid, opp[i] * n + cell, i * n + from_cell).reshape(-1)
    f64 = dict(dtype=torch.float64, device=dev)
    C, w = torch.tensor(c, **f64), torch.tensor(w, **f64)
    pairs = [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]
    CC = torch.stack([C[:, a] * C[:, b] for a, b in pairs])
    moments = torch.cat([torch.ones(1, Q, **f64), C.T, CC])
    twice = torch.tensor([1.0, 1, 1, 2, 2, 2], **f64)[:, None]
    eye = torch.tensor([1.0, 1, 1 if dim == 3 else 0, 0, 0, 0], **f64)[:, None]
    G = torch.tensor(g, **f64)[:, None]
    fluid = (~solid).reshape(-1)
    h = torch.zeros(Q, n, **f64)
    tau = torch.full((n,), 0.5 + 3.0 * (mu_p + m * sigma_y), **f64)

    def streamed():
        f = torch.take(h, src)
        mom = moments @ f
        return f, mom[0], mom[1:4], mom[4:]

    def velocity(d, j):
        return (j + 0.5 * (1 + d) * G) / (1 + d)

    def product(u, v):
        return torch.stack([0.5 * (u[a] * v[b] + u[b] * v[a]) for a, b in pairs])

    def even(d, rho, uu):      # w (d + rho (9/2 cc - 3/2 I) : uu), the even part of f_eq - w
        return w[:, None] * (d - 1.5 * rho * uu[:3].sum(0) + 4.5 * rho * (CC.T @ (twice * uu)))

    previous, residual, flow, checks = torch.zeros(3, n, **f64), -1.0, 0.0, 0
    for step in range(1, steps + 1):
        f, d, j, P = streamed()
        rho = 1 + d
        if check_every and step % check_every == 0:
            u = velocity(d, j)[:, fluid]
            if checks:
                residual = float(((u - previous).square().sum() / u.square().sum()).sqrt())
            previous, checks, flow = u, checks + 1, float(u[0].sum()) / mask.shape[2]
        if model == "IR":
            u = velocity(d, j)
            uu = product(u, u)
            T = P - d / 3 * eye - rho * uu
            norm = (twice * T * T).sum(0).sqrt()
            limit = math.sqrt(2.0) * sigma_y
            flows = (norm > 0) & (norm >= limit)
            safe = torch.where(flows, norm, torch.ones_like(norm))
            s = torch.where(flows, -(safe - limit) / (0.5 + 3 * mu_p) / safe, 0.0) * T
            sig = torch.where(flows, -(6 * mu_p * safe + limit) / (1 + 6 * mu_p) / safe, -1.0) * T
            A = -(sig - sig[:3].sum(0) / dim * eye) + 0.5 * s
            fs = 4.5 * w[:, None] * (CC.T @ (twice * A) - A[:3].sum(0) / 3)
            h = even(d, rho, uu) + fs + 3 * w[:, None] * (C @ (rho * (u + 0.5 * G)))
        else:
            u = j / rho
            uu = product(u, u)
            T = P - d / 3 * eye - rho * uu
            gd = 1.5 / tau * (2 * (twice * T * T).sum(0)).sqrt()
            y = sigma_y / rho
            low = mu_p + m * y
            at_c = mu_p - y * math.expm1(-m * gdot_c) / gdot_c
            above = mu_p - y * torch.expm1(-m * gd) / torch.where(gd > 0, gd, torch.ones_like(gd))
            nu = torch.where(gd >= gdot_c, above, (gdot_c - gd) / gdot_c * low + gd / gdot_c * at_c)
            tau = 0.5 + 3 * nu
            odd_tau = 0.5 + magic / (tau - 0.5)
            e = even(d, rho, uu)
            o = 3 * w[:, None] * (C @ (rho * u))
            plus, minus = 0.5 * (f + f[opp]), 0.5 * (f - f[opp])
            v = u + G
            h = (f - (plus - e) / tau - (minus - o) / odd_tau + even(d, rho, product(v, v)) - e
                 + 3 * w[:, None] * (C @ (rho * G)))
    _, d, j, _ = streamed()
    rho, u = (1 + d) * fluid, velocity(d, j) * fluid
    return rho, u, residual, flow


def exact(case, seed):
    if case["kind"] == "mix":
        got = {}
        for q in _mix(case, seed):
            rho, u, _, flow = _march(q["lattice"], q["model"], q["mask"], case["steps"],
                                     case["check_every"], **_params(q))
            g = got.setdefault(q["storage"], {"flow": [], "rho": [], "u": []})
            g["flow"].append(flow)
            g["rho"].append(rho)
            g["u"].append(u.reshape(-1))
        return {k: {"flow": np.array(g["flow"]), "rho": torch.cat(g["rho"]), "u": torch.cat(g["u"])}
                for k, g in got.items()}
    mask, p = _flow(case, seed)
    rho, u, residual, flow = _march(case["lattice"], case["model"], mask, case["steps"],
                                    case["check_every"], **p)
    return dict({"residual": residual, "flow": flow} if case["check_every"] else {}, rho=rho, u=u)
