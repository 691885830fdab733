"""The work that a user of the fire model has it do, as timed cases.

A case is one pass through the public entry points: a fire front carried some
steps on from a given state (a forecast from an analysis, a coupled model's
steps, an ensemble's cycle), or a gradient for data assimilation.  Every pass
starts from the same state, put back by fire_set_state as a program that
restarts from an analysis does, and ends with the whole state copied out.

Inputs follow the recipe of this repository's workloads: wind 5 m/s with
smooth 1.5 m/s perturbations of 300 m length, 20 Gaussian hills of slope up
to 0.4, 13 fuel classes on Voronoi patches of 30 m pixels, fires that have
burnt for some time.  `exact` is the same method in plain torch, 64 bits.
"""
import math

import numpy as np
import torch

import paper_1102_1343_gb300 as fire

T0 = 300.0        # model time of the starting states (s)
DX_ATM = 60.0     # atmospheric mesh of the recipe (m)
Z_F = 6.1         # height of the wind input (m)
Z_EXT = 50.0      # heat extinction depth (m)


def listed():
    run = dict(kind="run", sr=10, precision="fp32", dt=0.5, moisture=False, mult=False, plain=False)
    return [
        # the plain 600 m circle fire of the first configuration, all of its 120 steps: the
        # smallest mesh, where launches and latency are the time
        dict(run, name="circle100_fp64", nxa=10, nya=10, precision="fp64", steps=120, fires=1, radius=10.0, plain=True),
        # one step on buffers that a host framework owns, on a small ragged mesh
        dict(run, name="noalloc_230x170", kind="noalloc", nxa=23, nya=17, steps=1, fires=2, radius=60.0),
        # the steps of a coupled model: wind from the model levels, fire step, heat into the
        # tendencies; refinement 5 with an odd node count, per-node moisture and multiplier
        dict(run, name="coupled_815x585_nodes", kind="coupled", nxa=163, nya=117, sr=5, steps=12, fires=6, radius=80.0, moisture=True, mult=True),
        # the line-fire mesh of the second configuration, in both precisions
        dict(run, name="front2000_fp32", nxa=200, nya=200, steps=50, fires=3, radius=500.0),
        dict(run, name="front2000_fp64", nxa=200, nya=200, precision="fp64", steps=4, fires=3, radius=500.0),
        # the large mesh (820 atmospheric cells, 67 M nodes) with 50 small fires
        dict(run, name="points8200_fp32", nxa=820, nya=820, steps=12, fires=50, radius=100.0),
        # the same mesh two fifths burnt, each step called with host winds and host heat fluxes
        dict(run, name="burning8200_host", kind="host", nxa=820, nya=820, steps=6, fires=50, radius=3000.0),
        # drip torches at work: every step of the pass lies in their ignition windows
        dict(run, name="torches1400_fp32", kind="torches", nxa=140, nya=100, steps=20, fires=4, radius=30.0),
        # gradients: arrival times on the 510 x 510 assimilation mesh through the autograd
        # function (32-bit parameters, checkpoints), and in 64 bits with every state kept
        dict(run, name="adjoint510_fp32", kind="adjoint_fn", nxa=51, nya=51, steps=100, every=20, fires=1, radius=60.0),
        dict(run, name="adjoint510_fp64", kind="adjoint", nxa=51, nya=51, precision="fp64", steps=30, every=1, fires=1, radius=60.0),
        # the gradient of the heat misfit on a ragged mesh
        dict(run, name="adjoint_heat_370x290", kind="adjoint_heat", nxa=37, nya=29, steps=60, every=15, fires=1, radius=60.0),
        # an ensemble of uneven meshes, 40 steps of every member in one call
        dict(run, name="ensemble24_fp32", kind="ensemble", members=24, nxa=26, nya=130, steps=40, fires=1, radius=100.0),
    ]


def draw(rng):
    def size(lo, hi):  # spread over the logarithm
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["run", "run", "run", "noalloc", "coupled", "host", "torches", "adjoint_fn", "adjoint", "adjoint_heat",
                       "ensemble"])
    c = dict(kind=kind, sr=rng.choice([10, 10, 10, 4, 5, 7, 8, 12]), precision=rng.choice(["fp32", "fp32", "fp32", "fp64"]),
             dt=rng.choice([0.25, 0.5]), moisture=rng.random() < 0.25, mult=rng.random() < 0.25, plain=False,
             fires=rng.randint(1, 5), radius=float(rng.randint(15, 60)))
    if kind in ("adjoint_fn", "adjoint", "adjoint_heat"):
        c.update(nxa=size(12, 52), nya=size(12, 52), steps=rng.randint(10, 30), every=rng.choice([1, 5, 10, 20]), sr=rng.choice([5, 8, 10]),
                 precision="fp32" if kind != "adjoint" else c["precision"])
        if kind == "adjoint_fn":
            c.update(moisture=False, mult=False)  # its own parameters
    elif kind == "ensemble":
        c.update(members=rng.randint(2, 20), nxa=size(12, 26), nya=size(40, 120), steps=rng.randint(5, 30), fires=1, sr=10)
        if c["precision"] == "fp64":
            c.update(members=min(c["members"], 6), steps=rng.randint(2, 6), nya=min(c["nya"], 60))
    else:
        big = 60 if c["precision"] == "fp64" else 700 if kind in ("run", "host") else 200
        c.update(nxa=size(10, big), nya=size(10, big), steps=1 if kind == "noalloc" else rng.randint(2, 12))
        if kind == "host" or (kind == "run" and rng.random() < 0.4):
            c["radius"] = 0.2 * DX_ATM * min(c["nxa"], c["nya"])
    c["radius"] = float(round(min(c["radius"], 0.25 * DX_ATM * min(c["nxa"], c["nya"])), 1))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _classes(rng, plain):
    base = dict(windrf=0.36, weight=7.0, weight_is_tf=0.0, fgi=0.166, fueldepthm=0.305, savr=3500.0 / 0.3048, fuelmce=0.12,
                fueldens=32.0 * 0.45359237 / 0.3048 ** 3, st=0.0555, se=0.010, cmbcnst=18.608e6, fuelmc_g=0.08, chaparral=0.0)
    if plain:
        return [dict(base, fgi=0.5, weight=60.0, weight_is_tf=1.0)]
    return [dict(base, windrf=float(rng.uniform(0.1, 0.2)), weight=float(rng.uniform(7.0, 180.0)), fgi=float(rng.uniform(0.1, 2.0)),
                 fueldepthm=float(rng.uniform(0.3, 1.0)), savr=float(rng.uniform(1500.0, 2500.0)) / 0.3048,
                 fuelmce=float(rng.uniform(0.25, 0.40)), fuelmc_g=float(rng.uniform(0.04, 0.2))) for _ in range(13)]


def _smooth(rng, ny, nx, sigma):
    """White noise under a Gaussian of `sigma` cells, centred."""
    f = torch.as_tensor(rng.standard_normal((ny, nx)), device="cuda")
    for n, left in ((ny, True), (nx, False)):
        i = torch.arange(n, dtype=torch.float64, device="cuda")
        g = torch.exp(-(i[:, None] - i[None, :]) ** 2 / (2 * sigma * sigma))
        g = g / g.sum(1, keepdim=True)
        f = g @ f if left else f @ g.T
    return f - f.mean()


def _inputs(c, seed):
    """Every input of one mesh, on the GPU, in the context's precision."""
    rng = np.random.default_rng([1102, seed])
    nxa, nya, sr = c["nxa"], c["nya"], c["sr"]
    nx, ny, dx = nxa * sr, nya * sr, DX_ATM / sr
    T = torch.float64 if c["precision"] == "fp64" else torch.float32
    f64 = dict(dtype=torch.float64, device="cuda")
    p = dict(c=c, T=T, nx=nx, ny=ny, dx=dx, classes=_classes(rng, c["plain"]))
    x, y = (torch.arange(nx, **f64) + 0.5) * dx, (torch.arange(ny, **f64) + 0.5) * dx
    if c["plain"]:
        p.update(u=torch.full((nya, nxa + 1), 3.0, **f64), v=torch.zeros((nya + 1, nxa), **f64),
                 zx=torch.zeros((ny, nx), **f64), zy=torch.zeros((ny, nx), **f64), fuel=torch.zeros((ny, nx), dtype=torch.uint8, device="cuda"))
    else:
        for k, shape, mean in (("u", (nya, nxa + 1), 5.0), ("v", (nya + 1, nxa), 0.0)):
            w = _smooth(rng, *shape, 300.0 / DX_ATM)
            p[k] = mean + w * (1.5 / w.std().clamp_min(1e-12))
        hx, hy, s, h = (torch.as_tensor(rng.uniform(a, b, 20), **f64)[:, None] for a, b in ((0, nx * dx), (0, ny * dx), (200, 800), (0.5, 1)))
        ex, ey = torch.exp(-(x - hx) ** 2 / (2 * s * s)), torch.exp(-(y - hy) ** 2 / (2 * s * s))
        zx, zy = (ey * h).T @ (-(x - hx) / (s * s) * ex), (-(y - hy) / (s * s) * ey * h).T @ ex
        m = 0.4 / math.sqrt(float((zx * zx + zy * zy).max()))
        p.update(zx=zx * m, zy=zy * m)
        b = max(1, round(30.0 / dx))  # nodes of a 30 m data pixel
        cy, cx = -(-ny // b), -(-nx // b)
        site = torch.as_tensor(rng.uniform(0, 1, (400, 2)), dtype=torch.float32, device="cuda") * torch.tensor([cy, cx], device="cuda")
        cls = torch.as_tensor(rng.integers(0, 13, 400).astype(np.uint8), device="cuda")
        px = torch.arange(cx, dtype=torch.float32, device="cuda")
        rows = [cls[((torch.full((cx, 1), float(j), device="cuda") - site[:, 0]) ** 2 + (px[:, None] - site[:, 1]) ** 2).argmin(1)] for j in range(cy)]
        p["fuel"] = torch.stack(rows).repeat_interleave(b, 0)[:ny].repeat_interleave(b, 1)[:, :nx].contiguous()
    mf = torch.tensor([k["fuelmc_g"] for k in p["classes"]], **f64)
    p["moist"] = p["mult"] = None
    if c["moisture"] or c["kind"] == "adjoint_fn":
        f = torch.as_tensor(rng.uniform(-0.03, 0.03, (nya, nxa)), **f64).repeat_interleave(sr, 0).repeat_interleave(sr, 1)
        p["moist"] = (mf[p["fuel"].long()] + f).clamp_min(0.01)
    if c["mult"] or c["kind"] == "adjoint_fn":
        p["mult"] = 1 + 0.2 * torch.sin(2 * math.pi * x / 900.0 + rng.uniform(0, 6)) * torch.cos(2 * math.pi * y / 700.0)[:, None]
    for k in ("u", "v", "zx", "zy", "moist", "mult"):
        if p[k] is not None:
            p[k] = p[k].to(T).contiguous()
    # fires that have burnt since before T0, at least a quarter of the mesh away from its edges where there are few
    mx, my = (min(0.25 * n * dx, c["radius"] + 2000.0) for n in (nx, ny))
    at = [(0.5 * nx * dx, 0.5 * ny * dx)] if c["fires"] == 1 else \
         [(rng.uniform(mx, nx * dx - mx), rng.uniform(my, ny * dx - my)) for _ in range(c["fires"])]
    psi = torch.full((ny, nx), math.inf, **f64)
    for cx_, cy_ in at:
        psi = torch.minimum(psi, torch.sqrt((x - cx_) ** 2 + ((y - cy_) ** 2)[:, None]) - c["radius"] * rng.uniform(0.7, 1.0))
    psi = psi.to(T)
    tign = torch.where(psi <= 0, T0 + psi.double() / 0.5, torch.full((ny, nx), math.inf, **f64))
    tf = torch.tensor([_burn_time(k) for k in p["classes"]], **f64)[p["fuel"].long()]
    frac = torch.where(psi < 0, torch.exp(-(T0 - torch.where(psi <= 0, tign, torch.full_like(tign, T0))) / tf), torch.ones_like(tign)).to(T)
    p.update(psi=psi, tign=tign, frac=frac)
    if c["kind"] == "torches":  # started before the pass and still walking after it
        p["ign"] = [dict(ax=rng.uniform(0.3, 0.5) * nx * dx, ay=rng.uniform(0.3, 0.7) * ny * dx, bx=0.0, by=0.0, t_start=T0 - 30.3 - 7 * k, radius=12.0,
                         speed=0.4, vx=rng.uniform(0.8, 1.5), vy=rng.uniform(-1, 1), t_end=T0 + 60.0) for k in range(4)]
        for g in p["ign"]:
            g["bx"], g["by"] = g["ax"], g["ay"]
    if c["kind"] == "coupled":
        nz = 20
        k = torch.arange(nz + 1, **f64)[:, None, None]
        for name, shape in (("u", (nya, nxa + 1)), ("v", (nya + 1, nxa)), ("m", (nya, nxa))):
            zw = 3000.0 * (k / nz) ** 1.6 * (1 + 0.03 * torch.as_tensor(rng.standard_normal(shape), **f64))
            z = 0.5 * (zw[1:] + zw[:-1])
            if name == "m":
                p.update(zw=zw.contiguous(), rho=1.2 * torch.exp(-z / 8000.0), mu=9.0e4 * (1 + 0.02 * torch.as_tensor(rng.standard_normal(shape), **f64)))
                continue
            z0 = torch.as_tensor(rng.uniform(0.02, 0.5, shape), **f64)
            ref = p[name].double() / torch.log(Z_F / z0)  # a log profile through the recipe's wind
            p["w3" + name] = tuple(a.to(T).contiguous() for a in (ref * torch.log(z / z0), z, z0))
    if c["kind"].startswith("adjoint"):
        # observed arrival times a little off a smooth front, on nodes up to some distance ahead
        d = (psi.double() - 0).clamp_min(0)
        p["tobs"] = torch.where(psi < 40, T0 + d / 0.6 * (1 + 0.1 * torch.sin(x / 50.0)), torch.full_like(tign, math.nan))
        # observed heat release: up to 2 MJ/m^2 where it has burnt, noise elsewhere, a tenth of the cells unseen
        q = torch.as_tensor(rng.uniform(0.0, 2e6, (nya, nxa)), **f64) * torch.where(_cells(psi.double(), sr) < 0, 1.0, 1e-3)
        p["qobs"] = torch.where(torch.as_tensor(rng.uniform(0, 1, (nya, nxa)) < 0.9, device="cuda"), q, torch.full_like(q, math.nan))
    return p


def _members(c, seed):
    sizes = np.random.default_rng([c["nxa"], c["nya"], c["members"]]).integers(c["nxa"], c["nya"] + 1, c["members"])
    return [_inputs(dict(c, nxa=int(n), nya=int(n)), seed * 1000 + k) for k, n in enumerate(sizes)]


def _grid(p):
    c = p["c"]
    return fire.make_grid(c["nxa"], c["nya"], c["sr"], c["sr"], DX_ATM, DX_ATM, fire.FIRE_FP64 if c["precision"] == "fp64" else fire.FIRE_FP32)


def _model(p):
    c = p["c"]
    own = {} if c["kind"] == "adjoint_fn" else dict(mult=p["mult"], moisture=p["moist"])
    cpu = {k: None if a is None else a.cpu() for k, a in own.items()}
    m = fire.FireModel(c["nxa"], c["nya"], c["sr"], DX_ATM, p["classes"], p["fuel"].cpu(), p["zx"].cpu(), p["zy"].cpu(), p.get("ign", ()),
                       precision=c["precision"], **cpu)
    return m


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        ps = _members(case, seed)
        n = [p["nx"] * p["ny"] for p in ps]
        na = [p["c"]["nxa"] * p["c"]["nya"] for p in ps]
        f64 = dict(dtype=torch.float64, device="cuda")
        out = dict(psi=torch.empty(sum(n), dtype=ps[0]["T"], device="cuda"), tign=torch.empty(sum(n), **f64),
                   frac=torch.empty(sum(n), dtype=ps[0]["T"], device="cuda"), hs=torch.empty(sum(na), **f64), hl=torch.empty(sum(na), **f64))
        cut = {k: torch.split(a, na if k in ("hs", "hl") else n) for k, a in out.items()}
        torch.cuda.synchronize()
        ens = _Ensemble([dict(grid=_grid(p), classes=p["classes"], fuel_class_dev=p["fuel"], moisture_dev=p["moist"], spread_mult_dev=p["mult"],
                              dzdx_dev=p["zx"], dzdy_dev=p["zy"]) for p in ps])
        return dict(kind=kind, case=case, ens=ens, u=[p["u"] for p in ps], v=[p["v"] for p in ps], out=out, cut=cut,
                    state=[(p["psi"], p["tign"], p["frac"]) for p in ps])
    p = _inputs(case, seed)
    s = dict(kind=kind, case=case, p=p, u=p["u"], v=p["v"], state=(p["psi"], p["tign"], p["frac"]))
    f64 = dict(dtype=torch.float64, device="cuda")
    if kind == "noalloc":
        s.update(grid=_grid(p), psi=torch.empty_like(p["psi"]), frac=torch.empty_like(p["frac"]), tign=p["tign"].clone(),
                 hs=torch.empty((case["nya"], case["nxa"]), **f64), hl=torch.empty((case["nya"], case["nxa"]), **f64),
                 status=torch.zeros(1, dtype=torch.int32, device="cuda"))
        return s
    s["m"] = _model(p)
    s["out"] = dict(psi=torch.empty_like(p["psi"]), tign=torch.empty_like(p["tign"]), frac=torch.empty_like(p["frac"]))
    if kind == "host":
        s.update(u=p["u"].cpu().pin_memory(), v=p["v"].cpu().pin_memory(),
                 hs=torch.empty((case["nya"], case["nxa"]), dtype=torch.float64).pin_memory(),
                 hl=torch.empty((case["nya"], case["nxa"]), dtype=torch.float64).pin_memory())
    if kind == "coupled":
        s.update(u=torch.empty_like(p["u"]), v=torch.empty_like(p["v"]), rth=torch.zeros_like(p["rho"]), rqv=torch.zeros_like(p["rho"]))
    return s


class _Ensemble:
    """The handle, given back when the program drops it."""

    def __init__(self, members):
        self.h = fire.fire_ensemble_create(members, torch.cuda.current_stream().cuda_stream)
        self.ctx = [fire.fire_ensemble_member(self.h, k) for k in range(len(members))]

    def __del__(self):
        fire.fire_ensemble_destroy(self.h)


def run(state):
    s, kind, c = state, state["kind"], state["case"]
    dt, n = c["dt"], c["steps"]
    if kind == "ensemble":
        e, o = s["ens"], s["cut"]
        for ctx, st in zip(e.ctx, s["state"]):
            fire.fire_set_state(ctx, *st, T0)
        fire.fire_ensemble_step(e.h, n, dt, s["u"], s["v"], o["hs"], o["hl"])
        for k, ctx in enumerate(e.ctx):
            fire.fire_get_state(ctx, o["psi"][k], o["tign"][k], o["frac"][k])
        return s["out"]
    p = s["p"]
    if kind == "noalloc":
        fire.fire_step_noalloc(s["grid"], p["classes"], p["psi"], s["psi"], p["frac"], s["frac"], s["tign"], p["fuel"], p["mult"], p["zx"], p["zy"],
                               p["u"], p["v"], T0, dt, s["hs"], s["hl"], s["status"], torch.cuda.current_stream().cuda_stream)
        return {k: s[k] for k in ("psi", "tign", "frac", "hs", "hl")}
    m = s["m"]
    if kind == "adjoint_fn":
        par = [a.detach().requires_grad_() for a in (p["mult"], p["moist"], p["u"], p["v"])]
        J = fire.FireAdjointFn.apply(m, (*s["state"], T0), *par, p["tobs"], dt, n, c["every"])
        return dict(J=J.detach(), grads=torch.autograd.grad(J, par))
    m.set_state(*s["state"], T0)
    if kind in ("adjoint", "adjoint_heat"):
        J, *g = m.adjoint(s["u"], s["v"], dt, n, p["tobs"], c["every"]) if kind == "adjoint" else \
            m.adjoint_heat(s["u"], s["v"], dt, n, p["qobs"], c["every"])
        return dict(J=J, grads=[a.to(p["T"]) for a in g])  # as the controls of the assimilation are held
    if kind == "host":
        for _ in range(n):
            fire.fire_step_host(m.ctx, s["u"], s["v"], dt, s["hs"], s["hl"])
        hs, hl = s["hs"], s["hl"]
    elif kind == "coupled":
        for _ in range(n):
            for k in ("u", "v"):
                fire.fire_wind_at_height(*p["w3" + k], Z_F, s[k])
            hs, hl = m.step(s["u"], s["v"], dt)
            s["rth"].zero_()
            s["rqv"].zero_()
            fire.fire_heat_insertion(hs, hl, p["zw"], p["rho"], p["mu"], Z_EXT, s["rth"], s["rqv"])
    else:
        hs, hl = m.run(n, s["u"], s["v"], dt)
    o = s["out"]
    fire.fire_get_state(m.ctx, o["psi"], o["tign"], o["frac"])
    out = dict(o, hs=hs, hl=hl)
    if kind == "coupled":
        out.update(u=s["u"], v=s["v"], rth=s["rth"], rqv=s["rqv"])
    return out


def work(case):
    """Per node and step: psi and F read and written, fuel class, slopes, and t_i (a double, read where the node burns; counted
    everywhere), about 160 operations.  A gradient: the forward states again, lambda in and out and four sums in and out."""
    w = 8 if case["precision"] == "fp64" else 4
    step = 4 * w + 2 * w + 1 + 8 + (w if case["mult"] or case["kind"] == "adjoint_fn" else 0) + (3 * w if case["moisture"] or case["kind"] == "adjoint_fn" else 0)
    if case["kind"] == "ensemble":
        lo, hi = case["nxa"], case["nya"]
        nodes = case["members"] * case["sr"] ** 2 * sum(k * k for k in range(lo, hi + 1)) / (hi - lo + 1)
    else:
        nodes = case["nxa"] * case["nya"] * case["sr"] ** 2
    flops = 160.0
    extra = 2 * (2 * w + 8) if case["kind"] != "noalloc" else 0  # the state put back and copied out, once
    if case["kind"].startswith("adjoint"):
        step += 4 * w + 24 + 5 * w + 1 + 2 * 4 * 8
        flops += 500.0
    return {"bytes": nodes * (case["steps"] * step + extra), "flops": nodes * case["steps"] * flops}


# ---------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------
def _burn_time(k):
    return k["weight"] if k["weight_is_tf"] else -600.0 * k["weight"] / (1000.0 * math.log(0.6))


def _coefficients(p, moist):
    """R0, b, c, d, T_f, H_s, H_q per node (Rothermel's chain in English units), at the moisture field."""
    f64 = dict(dtype=torch.float64, device="cuda")
    g = {k: torch.tensor([float(a[k]) for a in p["classes"]], **f64)[p["fuel"].long()] for k in p["classes"][0]}
    ft, lb, btu = 0.3048, 0.45359237, 1055.05585262
    sig, load, dep = g["savr"] * ft, g["fgi"] * ft * ft / lb, g["fueldepthm"] / ft
    rho, heat = g["fueldens"] * ft ** 3 / lb, g["cmbcnst"] * lb / btu
    w0 = load / (1 + moist)
    rhob = w0 / dep
    beta = rhob / rho
    rel = beta / (3.348 * sig ** -0.8189)
    gmax = sig ** 1.5 / (495 + 0.0594 * sig ** 1.5)
    A = 1 / (4.77 * sig ** 0.1 - 7.27)
    x = moist / g["fuelmce"]
    eta = (1 - 2.59 * x + 5.11 * x * x - 3.52 * x ** 3).clamp(max=1.0)
    eta = torch.where((x >= 1) | (eta < 0), torch.zeros_like(eta), eta)
    IR = gmax * rel ** A * torch.exp(A * (1 - rel)) * w0 / (1 + g["st"]) * heat * eta * 0.174 * g["se"] ** -0.19
    xi = torch.exp((0.792 + 0.681 * sig.sqrt()) * (beta + 0.1)) / (192 + 0.2595 * sig)
    R0 = IR * xi / (rhob * torch.exp(-138 / sig) * (250 + 1116 * moist)) * ft / 60
    B, C, E = 0.02526 * sig ** 0.54, 7.47 * torch.exp(-0.133 * sig ** 0.55), 0.715 * torch.exp(-3.59e-4 * sig)
    c = R0 * C * (g["windrf"] * 60 / ft) ** B * rel ** -E
    tf = torch.tensor([_burn_time(a) for a in p["classes"]], **f64)[p["fuel"].long()]
    return dict(R0=R0, b=B, c=c, d=R0 * 5.275 * beta ** -0.3, tf=tf, Hs=g["fgi"] * g["cmbcnst"] / (1 + moist),
                Hq=(moist + 0.56) / (1 + moist) * 2.5e6 * g["fgi"])


def _nodes(w, sr, nx, ny, ux, uy):
    """Bilinear from the staggered points to the nodes; `ux`, `uy`: whether the points lie at cell centres along x, y."""
    def weights(n, pts, centred):
        f = ((torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / sr - (0.5 if centred else 0.0)).clamp(0, pts - 1)
        k = f.floor().clamp(max=max(pts - 2, 0)).long()
        return k, (k + 1).clamp(max=pts - 1), f - k
    i0, i1, a = weights(nx, w.shape[1], ux)
    j0, j1, b = weights(ny, w.shape[0], uy)
    r = w[:, i0] * (1 - a) + w[:, i1] * a
    return r[j0] * (1 - b)[:, None] + r[j1] * b[:, None]


def _ghost(a, b):
    g = a + (a - b)
    g = torch.where(a > g, a, g)
    return torch.where(b > g, b, g)


def _pad(f):
    f = torch.cat([_ghost(f[:, :1], f[:, 1:2]), f, _ghost(f[:, -1:], f[:, -2:-1])], 1)
    return torch.cat([_ghost(f[:1], f[1:2]), f, _ghost(f[-1:], f[-2:-1])], 0)


def _rate(p, f, q):
    """dpsi/dt: Godunov gradient, normal from central differences (zero where they are rounding), eps S Lap."""
    zero = torch.zeros((), dtype=torch.float64, device="cuda")
    one = torch.ones_like(zero)
    dx, g = p["dx"], _pad(f)
    l, r, d, u = g[1:-1, :-2], g[1:-1, 2:], g[:-2, 1:-1], g[2:, 1:-1]
    tau = 1e-9 if p["T"] == torch.float64 else 1e-6

    def up(a, b):
        m, n = torch.where(a > 0, a, zero), torch.where(b < 0, b, zero)
        return torch.where(m * m > n * n, m, n)
    xm, xp, ym, yp = (f - l) / dx, (r - f) / dx, (f - d) / dx, (u - f) / dx
    gx, gy = up(xm, xp), up(ym, yp)
    g2 = gx * gx + gy * gy
    grad = torch.where(g2 > 0, torch.sqrt(torch.where(g2 > 0, g2, one)), zero)
    cx, cy = (torch.where((a - b).abs() <= tau * (a.abs() + b.abs()), zero, (a - b) / (2 * dx)) for a, b in ((r, l), (u, d)))
    n2 = cx * cx + cy * cy
    rn = torch.where(n2 > 0, 1 / torch.sqrt(torch.where(n2 > 0, n2, one)), zero)
    U, tp = (q["un"] * cx + q["vn"] * cy) * rn, (q["zx"] * cx + q["zy"] * cy) * rn
    on = U > 0
    pw = torch.where(on, torch.where(on, U.clamp(max=30.0), one) ** q["b"], zero)
    t = torch.where(tp > 0, tp, zero)
    S = q["m"] * (q["R0"] + q["c"] * pw + q["d"] * t * t).clamp_min(0)
    return -S * grad + p["c"].get("eps", 0.4) * S * ((xp - xm) + (yp - ym))


def _heun(p, f, dt, q):
    k1 = _rate(p, f, q)
    return f + dt * (0.5 * k1 + 0.5 * _rate(p, f + dt * k1, q))


def _crossed(f, new, tign, t, dt):
    hit = (f > 0) & (new <= 0) & torch.isinf(tign)
    den = torch.where(hit, f - new, torch.ones_like(f))
    return torch.where(hit, t + f * dt / den, tign)


def _fraction(f, tign, t, tf):
    """Fuel fraction: four subcells of cell centre, edge midpoints and corner."""
    zero = torch.zeros((), dtype=torch.float64, device="cuda")
    D = torch.where(f < 0, t - torch.where(f < 0, tign, torch.full_like(tign, t)), zero)
    P = _pad(f)
    D = torch.cat([D[:, :1], D, D[:, -1:]], 1)
    D = torch.cat([D[:1], D, D[-1:]], 0)
    D = torch.where(P >= 0, zero, D)

    def at(a, i, j):
        return a[1 + j:a.shape[0] - 1 + j, 1 + i:a.shape[1] - 1 + i]
    burnt = 0.0
    for i in (-1, 1):
        for j in (-1, 1):
            sp = sa = sd = 0.0
            for pts in (((0, 0),), ((0, 0), (i, 0)), ((0, 0), (0, j)), ((0, 0), (i, 0), (0, j), (i, j))):
                v = sum(at(P, *k) for k in pts) / len(pts)
                sp, sa = sp + v, sa + v.abs()
                sd = sd + torch.where(v >= 0, zero, sum(at(D, *k) for k in pts) / len(pts))
            beta = torch.where(sa > 0, 0.5 * (1 - sp / torch.where(sa > 0, sa, torch.ones_like(sa))), zero)
            burnt = burnt + beta * (1 - torch.exp(-0.25 * sd / tf))
    return 1 - 0.25 * burnt


def _torch_lines(p, f, tign, t):
    x = (torch.arange(p["nx"], dtype=torch.float64, device="cuda") + 0.5) * p["dx"]
    y = ((torch.arange(p["ny"], dtype=torch.float64, device="cuda") + 0.5) * p["dx"])[:, None]
    for g in p.get("ign", ()):
        if not g["t_start"] <= t <= g["t_end"] + g["radius"] / g["speed"]:
            continue
        tt = min(t, g["t_end"])
        sx, sy = g["vx"] * (tt - g["t_start"]), g["vy"] * (tt - g["t_start"])
        rho, L2 = min(g["radius"], g["speed"] * (t - g["t_start"])), sx * sx + sy * sy
        a = (((x - g["ax"]) * sx + (y - g["ay"]) * sy) / L2).clamp(0, 1) if L2 > 0 else torch.zeros_like(f)
        d = torch.sqrt((x - g["ax"] - a * sx) ** 2 + (y - g["ay"] - a * sy) ** 2)
        hit = (f > 0) & (d - rho <= 0) & torch.isinf(tign)
        tign = torch.where(hit, (g["t_start"] + a * (tt - g["t_start"]) + d / g["speed"]).clamp(max=t), tign)
        f = torch.minimum(f, d - rho)
    return f, tign


def _cells(a, sr):
    return a.reshape(a.shape[0] // sr, sr, a.shape[1] // sr, sr).mean((1, 3))


def _fields(p, u, v):
    c = p["c"]
    moist = p["moist"].double() if p["moist"] is not None else torch.tensor([k["fuelmc_g"] for k in p["classes"]], dtype=torch.float64,
                                                                          device="cuda")[p["fuel"].long()]
    q = dict(zx=p["zx"].double(), zy=p["zy"].double(), m=p["mult"].double() if p["mult"] is not None else torch.ones((), dtype=torch.float64, device="cuda"))
    q.update(_coefficients(p, moist))
    q.update(un=_nodes(u, c["sr"], p["nx"], p["ny"], False, True), vn=_nodes(v, c["sr"], p["nx"], p["ny"], True, False))
    return q


def _level(prof):
    """The wind at Z_F: linear in ln z through (z0, 0) and the levels."""
    w, z, z0 = (a.double() for a in prof)
    x, out = math.log(Z_F), None
    xl, ul = torch.log(z0), torch.zeros_like(z0)
    out, found = torch.zeros_like(z0), torch.zeros_like(z0, dtype=torch.bool)
    for k in range(z.shape[0]):
        ok, xk = z[k] > z0, torch.log(z[k].clamp_min(1e-30))
        here = ok & ~found & (x <= xk)
        out = torch.where(here, ul + (w[k] - ul) * (x - xl) / torch.where(here, xk - xl, torch.ones_like(xk)), out)
        found = found | here
        xl, ul = torch.where(ok, xk, xl), torch.where(ok, w[k], ul)
    return torch.where(Z_F > z0, torch.where(found, out, ul), torch.zeros_like(z0))


def _forward(p):
    c, sr, dt = p["c"], p["c"]["sr"], p["c"]["dt"]
    u, v = (_level(p["w3u"]), _level(p["w3v"])) if c["kind"] == "coupled" else (p["u"].double(), p["v"].double())
    q = _fields(p, u, v)
    f, tign, F, t = p["psi"].double(), p["tign"], p["frac"].double(), T0
    for _ in range(c["steps"]):
        f, tign = _torch_lines(p, f, tign, t)
        new = _heun(p, f, dt, q)
        tign = _crossed(f, new, tign, t, dt)
        f, t = new, t + dt
        F0, F = F, _fraction(f, tign, t, q["tf"])
    out = dict(psi=f, tign=tign, frac=F, hs=_cells((F0 - F) * q["Hs"], sr) / dt, hl=_cells((F0 - F) * q["Hq"], sr) / dt)
    if c["kind"] == "coupled":
        zw = p["zw"]
        S = (torch.exp(-zw[:-1] / Z_EXT) - torch.exp(-zw[1:] / Z_EXT)) / (zw[1:] - zw[:-1])
        out.update(u=u, v=v, rth=p["mu"] * out["hs"] / (1004.0 * p["rho"]) * S, rqv=p["mu"] * out["hl"] / (2.5e6 * p["rho"]) * S)
    return out


def _gradient(p):
    """J and its gradients by torch's reverse mode, one step at a time."""
    c, sr, dt, heat = p["c"], p["c"]["sr"], p["c"]["dt"], p["c"]["kind"] == "adjoint_heat"
    moist = p["moist"].double() if p["moist"] is not None else torch.tensor([k["fuelmc_g"] for k in p["classes"]], dtype=torch.float64,
                                                                          device="cuda")[p["fuel"].long()]
    mult = p["mult"].double() if p["mult"] is not None else torch.ones_like(moist)
    par = [a.clone().requires_grad_() for a in (mult, moist, p["u"].double(), p["v"].double())]
    q = dict(_fields(p, p["u"].double(), p["v"].double()))
    names = ("R0", "c", "d", "m", "un", "vn")
    co = _coefficients(p, par[1])
    live = dict(R0=co["R0"], c=co["c"], d=co["d"], m=par[0] * 1.0, un=_nodes(par[2], sr, p["nx"], p["ny"], False, True),
                vn=_nodes(par[3], sr, p["nx"], p["ny"], True, False))
    for k in names:
        q[k] = live[k].detach()
    states, times, tign = [p["psi"].double()], [T0], p["tign"]
    for _ in range(c["steps"]):
        new = _heun(p, states[-1], dt, q)
        tign = _crossed(states[-1], new, tign, times[-1], dt)
        states.append(new)
        times.append(times[-1] + dt)
    set_now = torch.isfinite(tign) & torch.isinf(p["tign"])
    lam = torch.zeros_like(states[0])
    sums = {k: torch.zeros_like(q[k]) for k in names}
    gm = torch.zeros_like(moist)
    if heat:
        f, tg, hs = states[-1].clone().requires_grad_(), tign.clone().requires_grad_(), _coefficients(p, moist)["Hs"].clone().requires_grad_()
        F = _fraction(f, tg, times[-1], q["tf"])
        Q = _cells((p["frac"].double() - F) * hs, sr)
        see = torch.isfinite(p["qobs"])
        J = 0.5 * (torch.where(see, Q - torch.where(see, p["qobs"], torch.zeros_like(Q)), torch.zeros_like(Q)) ** 2).sum()
        lam, seed, ghs = torch.autograd.grad(J, (f, tg, hs))
        gm = torch.autograd.grad(_coefficients(p, par[1])["Hs"], par[1], ghs)[0]
        seed = torch.where(torch.isfinite(seed), seed, torch.zeros_like(seed))
    else:
        see = torch.isfinite(tign) & torch.isfinite(p["tobs"])
        seed = torch.where(see, tign - torch.where(see, p["tobs"], tign), torch.zeros_like(tign))
        seed = torch.where(see, seed, torch.zeros_like(seed))
        J = 0.5 * (seed ** 2).sum()
    for s in range(c["steps"] - 1, -1, -1):
        f = states[s].clone().requires_grad_()
        w = {k: q[k].clone().requires_grad_() for k in names}
        new = _heun(p, f, dt, dict(q, **w))
        hit = (states[s] > 0) & (states[s + 1] <= 0) & set_now & (tign >= times[s]) & (tign <= times[s + 1])
        ti = torch.where(hit, f * dt / torch.where(hit, f - new, torch.ones_like(f)), torch.zeros_like(f))
        lam, *g = torch.autograd.grad((lam * new).sum() + (torch.where(hit, seed, torch.zeros_like(seed)) * ti).sum(), [f] + [w[k] for k in names])
        for k, a in zip(names, g):
            sums[k] += a
    g = torch.autograd.grad([live[k] for k in names], par, [sums[k] for k in names])
    return dict(J=float(J), grads=[g[0], g[1] + gm, g[2], g[3]])


def exact(case, seed):
    if case["kind"] == "ensemble":
        got = [_forward(p) for p in _members(case, seed)]
        return {k: torch.cat([o[k].reshape(-1) for o in got]) for k in ("psi", "tign", "frac", "hs", "hl")}
    p = _inputs(case, seed)
    if not case["kind"].startswith("adjoint"):
        return _forward(p)
    out = _gradient(p)
    if case["kind"] == "adjoint_fn":
        out["grads"] = tuple(out["grads"])
    return out
