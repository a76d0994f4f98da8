"""What a user of this library has it do, as timed cases.

Every case goes through the public Python entry points (the C ABI's names,
and the autograd functions for gradients).  Inputs are made on the GPU from
the seed; what is set up once per problem (context, angle grid, metric, time
step) is made beside them, as a program that steps many times keeps it.

Kinds of case ("do"):
  step     one RK2 step (rad_step) of a resident problem, and the moments of
           the result where "moments" names a method: the time loop's body
  groups   one multigroup RK2 step
  block    one RK2 step of a block that shares its x1 faces (with itself):
           halo packs and the two stages, as a decomposed domain steps
  moments  rad_moments alone: an analysis pass over a stored intensity
  grad     forward steps, the outgoing-flux loss and the backward pass
           through torch.autograd, with all gradients

Metrics: "cart" flat Cartesian, "sph" flat spherical, "ks" Kerr-Schild.
Angle grids: geodesic "level", or n_zeta x n_psi where "n_zeta" is set.
"""
import math

import numpy as np
import torch

import paper_2302_04283_gb300 as rad
from paper_2302_04283_gb300 import autograd as rag

DEV = "cuda"
RECON = {"dc": rad.RAD_RECON_DC, "plm": rad.RAD_RECON_PLM, "ppm": rad.RAD_RECON_PPM, "mapr": rad.RAD_RECON_MAPR}
COUPLE = {"thermal": rad.RAD_COUPLE_THERMAL, "emissivity": rad.RAD_COUPLE_EMISSIVITY, "none": rad.RAD_COUPLE_NONE}
FRAME = {"tetrad": rad.RAD_FRAME_TETRAD, "coord": rad.RAD_FRAME_COORD, "fluid": rad.RAD_FRAME_FLUID}
GAMMA = 5.0 / 3.0

DEFAULT = {"metric": "cart", "spin": 0.0, "level": 4, "n_zeta": 0, "n_psi": 0, "prec": "f32", "recon": "plm",
           "recon_ang": "dc", "coupling": "thermal", "gas": "turb", "bc": "periodic", "src": False, "moments": "",
           "frame": "tetrad", "tau": 0.0, "rad_dom": False, "groups": 0, "steps": 1}


def listed():
    return [
        # the smallest call: the paper's 2D hot spot (32 x 32 cells, 42 bins) in plain FP64, where launches and
        # the host path count
        {"name": "hotspot2d_f64", "do": "step", "n1": 32, "n2": 32, "n3": 1, "level": 2, "prec": "f64",
         "gas": "hotspot"},
        # the benchmark workload: turbulent gas in flat space, FP32 transport, tensor-core moments, gas source
        {"name": "turb3d_f32", "do": "step", "n1": 128, "n2": 128, "n3": 128, "level": 4, "prec": "f32",
         "src": True, "moments": "bf16"},
        # the same problem in plain FP64 (the library's default precision), at 64^3 cells
        {"name": "turb3d_f64", "do": "step", "n1": 64, "n2": 64, "n3": 64, "level": 4, "prec": "f64", "src": True,
         "moments": "simt"},
        # a torus around a spinning black hole at the paper's angular resolution, FP32, moments in the
        # coordinate frame (what a GRMHD solver takes)
        {"name": "torus3d_f32", "do": "step", "metric": "ks", "spin": 0.9, "n1": 128, "n2": 64, "n3": 64,
         "level": 6, "prec": "f32", "gas": "torus", "src": True, "moments": "bf16", "frame": "coord"},
        # the largest: 192 x 96 x 96 cells with 642 bins, moving torus gas with scattering
        {"name": "torus3d_big_f32", "do": "step", "metric": "ks", "spin": 0.9, "n1": 192, "n2": 96, "n3": 96,
         "level": 8, "prec": "f32", "gas": "torus_moving", "src": True, "moments": "bf16"},
        # a Kerr-Schild run in the default precision on a ragged grid
        {"name": "kerr3d_f64", "do": "step", "metric": "ks", "spin": 0.9, "n1": 61, "n2": 37, "n3": 34, "level": 3,
         "prec": "f64", "gas": "torus_moving", "src": True},
        # spherical flat space with the latitude-longitude angle grid (8 x 16, as in the paper's CPU timings) and
        # line reconstruction of the angular fluxes
        {"name": "latlong_f32", "do": "step", "metric": "sph", "n1": 90, "n2": 50, "n3": 44, "n_zeta": 8,
         "n_psi": 16, "prec": "f32", "recon_ang": "plm", "gas": "torus"},
        # multigroup transport with redshift between the groups, fixed emissivity
        {"name": "groups_f32", "do": "groups", "metric": "ks", "spin": 0.5, "n1": 48, "n2": 32, "n3": 30,
         "level": 3, "prec": "f32", "coupling": "emissivity", "groups": 6, "src": True},
        # one block of a domain split along x1 (each rank of a decomposed run does this between its exchanges)
        {"name": "block_f32", "do": "block", "n1": 72, "n2": 64, "n3": 81, "level": 4, "prec": "f32", "src": True},
        # an analysis pass: fluid-frame moments of a stored intensity, odd sizes
        {"name": "moments_fluid_f32", "do": "moments", "n1": 101, "n2": 67, "n3": 53, "level": 5, "prec": "f32",
         "moments": "bf16", "frame": "fluid"},
        # gradients of the outgoing flux in the opacities and the emissivity, axisymmetric Kerr-Schild, FP64
        {"name": "adjoint2d_f64", "do": "grad", "metric": "ks", "spin": 0.5, "n1": 256, "n2": 128, "n3": 1,
         "level": 4, "prec": "f64", "coupling": "emissivity", "gas": "smooth", "steps": 2},
        # gradients through the thermal coupling of a 3D flat problem, FP32, outflow along x1
        {"name": "adjoint3d_thermal_f32", "do": "grad", "n1": 45, "n2": 38, "n3": 33, "level": 4, "prec": "f32",
         "bc": "outflow", "steps": 1},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges."""
    do = rng.choice(["step", "step", "step", "step", "groups", "block", "moments", "grad"])
    c = {"do": do, "prec": rng.choice(["f32", "f32", "f64"])}
    if do == "block" or (do in ("step", "moments", "grad") and rng.random() < 0.5):
        c["metric"] = "cart"
    else:
        c["metric"] = rng.choice(["ks", "ks", "sph"])
        c["spin"] = round(rng.uniform(0.0, 0.95), 2) if c["metric"] == "ks" else 0.0
    if c["metric"] != "cart" and do == "step" and rng.random() < 0.3:
        c["n_zeta"], c["n_psi"] = rng.choice([4, 6, 8, 11]), 2 * rng.randint(4, 9)
        c["recon_ang"] = rng.choice(["dc", "plm"])
        bins = c["n_zeta"] * c["n_psi"]
    else:
        c["level"] = rng.choice([2, 3, 4, 4, 5, 6, 7, 8] if c["prec"] == "f32" and do != "grad" else [2, 3, 4, 4, 5])
        bins = 10 * c["level"] ** 2 + 2
        if c["metric"] == "ks" and do == "step" and rng.random() < 0.15:
            c["recon_ang"] = "mapr"
    # cells from a budget of cell-angles, spread over its logarithm
    most = {"step": 3e8, "groups": 4e7, "block": 1e8, "moments": 3e8, "grad": 8e6}[do]
    if c["prec"] == "f64":
        most /= 1 if do == "moments" else 8
    budget = math.exp(rng.uniform(math.log(4e4), math.log(most))) / bins
    groups = rng.randint(2, 8) if do == "groups" else 0
    if groups:
        c["groups"] = groups
        budget /= groups
    flat2 = do in ("step", "grad") and rng.random() < 0.3
    side = max(4.0, budget ** (0.5 if flat2 else 1.0 / 3.0))
    cap = 512 if flat2 else 160
    a, b = (min(cap, max(4, int(side * rng.uniform(0.6, 1.6)))) for _ in range(2))
    n3 = 1 if flat2 else min(cap, max(4, int(budget / (a * b))))
    if n3 > 1 and c["metric"] != "cart":
        n3 += n3 % 2
    c.update(n1=a, n2=b, n3=n3)
    if do == "groups":
        c["coupling"] = "emissivity"
    elif do != "moments":
        c["coupling"] = rng.choice(["thermal", "thermal", "thermal", "emissivity"] + (["none"] if do == "step" else []))
    if do == "step":
        c["recon"] = rng.choice(["plm", "plm", "plm", "plm", "dc", "ppm"])
        if c["coupling"] == "thermal" and rng.random() < 0.1:
            c["rad_dom"] = True
        elif rng.random() < 0.1:
            c["tau"] = 5.0
    if do in ("step", "groups", "block"):
        c["src"] = rng.random() < 0.7
    if do == "moments" or (do == "step" and rng.random() < 0.6):
        c["moments"] = "simt" if c["prec"] == "f64" else rng.choice(["bf16", "bf16", "simt"])
        c["frame"] = rng.choice(["tetrad", "coord", "fluid"])
    c["gas"] = "turb" if c["metric"] == "cart" else rng.choice(["torus", "torus_moving", "smooth"])
    if c["metric"] == "cart" and do in ("step", "grad"):
        c["bc"] = "outflow" if do == "grad" else rng.choice(["periodic", "outflow"])
    if do == "grad":
        c["steps"] = rng.choice([1, 2])
    return c


def _n_ang(c):
    return c["n_zeta"] * c["n_psi"] if c["n_zeta"] else 10 * c["level"] ** 2 + 2


def work(case):
    """Each input read once and each output written once; operations of the scheme as printed (per bin and stage
    about 14 per flux dimension with a limited slope, 26 for angular fluxes, 40 for the coupling)."""
    c = {**DEFAULT, **case}
    esz = 4 if c["prec"] == "f32" else 8
    cells = c["n1"] * c["n2"] * c["n3"]
    bins, g = cells * _n_ang(c), max(1, c["groups"])
    ndim = 3 if c["n3"] > 1 else 2
    per_stage = 14 * ndim + (26 if c["metric"] != "cart" else 0) + (40 if c["coupling"] != "none" else 0)
    mom = (bins * 20, cells * 10 * esz) if c["moments"] else (0, 0)
    gas = 8 * (7 + g * (2 + (1 if c["coupling"] == "emissivity" else 0)))
    if c["do"] == "moments":
        return {"bytes": bins * esz + mom[1] + (24 * cells if c["frame"] == "fluid" else 0), "flops": mom[0]}
    if c["do"] == "grad":
        # forward, and per step the recomputation and two reverse sweeps; state and gradients in and out
        return {"bytes": bins * esz * 2 + cells * 8 * (7 + 4), "flops": c["steps"] * bins * per_stage * 2 * 4}
    return {"bytes": 2 * bins * g * esz + cells * gas + (32 * cells * g if c["src"] else 0) + mom[1],
            "flops": bins * g * per_stage * 2 + mom[0]}


# ---------------------------------------------------------------- inputs

def _faces(c):
    n1, n2, n3 = c["n1"], c["n2"], c["n3"]
    if c["metric"] == "cart":
        return [np.linspace(0.0, 1.0, n + 1) for n in (n1, n2, n3)]
    return [np.exp(np.linspace(math.log(1.5 if c["metric"] == "ks" and c["spin"] > 0.6 else 2.0), math.log(50.0),
                               n1 + 1)),
            np.linspace(0.0, math.pi, n2 + 1), np.linspace(0.0, 2.0 * math.pi, n3 + 1)]


def _bc(c):
    if c["do"] == "block":
        return (("halo", "halo"), ("periodic", "periodic"), ("periodic", "periodic"))
    if c["metric"] != "cart":
        return (("outflow", "outflow"), ("polar", "polar"), ("periodic", "periodic"))
    if c["bc"] == "outflow":
        return (("outflow", "outflow"), ("periodic", "periodic"), ("periodic", "periodic"))
    return (("periodic", "periodic"),) * 3


def _inputs(c, seed, n_ang, nap, xf):
    """Gas fields (FP64) and the padded intensity of the case, on the GPU."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    sh = (c["n3"], c["n2"], c["n1"])
    f64 = dict(dtype=torch.float64, device=DEV)

    def uni(lo, hi, *shape):
        return torch.rand(shape, generator=g, **f64) * (hi - lo) + lo

    xc = [torch.tensor(0.5 * (x[1:] + x[:-1]), **f64) for x in xf]
    Z, Y, X = torch.meshgrid(xc[2], xc[1], xc[0], indexing="ij")

    def velocity(vmax):
        v = torch.zeros(sh + (3,), **f64)
        span = [float(x[-1] - x[0]) for x in xf]
        for comp in range(3):
            amp = torch.randn(27, generator=g, **f64).tolist()
            ph = uni(0.0, 2.0 * math.pi, 27).tolist()
            for m in range(27):
                k = (m % 3 + 1, m // 3 % 3 + 1, m // 9 + 1)
                v[..., comp] += amp[m] * torch.sin(2.0 * math.pi * (k[0] * X / span[0] + k[1] * Y / span[1]
                                                                    + k[2] * Z / span[2]) + ph[m])
        v *= vmax / v.square().sum(-1).sqrt().max()
        return (v / (1.0 - v.square().sum(-1, keepdim=True)).sqrt()).contiguous()

    def smooth():
        s = torch.zeros(sh, **f64)
        lx = (X.log() - xc[0][0].log()) / (xc[0][-1] / xc[0][0]).log() if c["metric"] != "cart" else X
        for m in (1, 2, 3):
            for n in (1, 2, 3):
                a, p = float(torch.randn(1, generator=g, **f64)), float(uni(0.0, 2.0 * math.pi, 1))
                s += a * torch.cos(2.0 * math.pi * m * lx + p) * torch.cos(2.0 * n * Y)
        return 2.0 * (s - s.min()) / (s.max() - s.min()) - 1.0

    gas = {"rho": torch.ones(sh, **f64), "u": torch.zeros(sh + (3,), **f64), "eta": None, "T": torch.ones(sh, **f64)}
    if c["gas"] == "hotspot":
        d2 = ((X - 0.5) * c["n1"]) ** 2 + ((Y - 0.5) * c["n2"]) ** 2
        gas["T"] = 1.0 + 2.0 * torch.exp(-d2 / 32.0)
        gas["alpha_a"], gas["alpha_s"] = torch.ones(sh, **f64), torch.zeros(sh, **f64)
    elif c["gas"] == "turb":
        gas["u"] = velocity(0.5)
        gas["alpha_a"], gas["alpha_s"] = 10.0 ** uni(-2.0, 2.0, *sh), 10.0 ** uni(-2.0, 2.0, *sh)
        gas["T"] = torch.exp(uni(math.log(0.5), math.log(2.0), *sh))
    elif c["gas"] == "smooth":
        gas["alpha_a"], gas["alpha_s"] = 10.0 ** smooth(), 10.0 ** smooth()
    else:
        rho = torch.exp(-((X - 10.0) ** 2 + (10.0 * torch.cos(Y)) ** 2) / 8.0) + 1e-4
        gas["rho"], gas["alpha_a"] = rho, rho.clone()
        moving = c["gas"] == "torus_moving"
        gas["alpha_s"] = 0.5 * rho if moving else torch.zeros(sh, **f64)
        if moving:
            gas["u"] = velocity(0.3)
    if c["coupling"] == "emissivity":
        gas["eta"] = 10.0 ** smooth() / (4.0 * math.pi) if c["gas"] == "smooth" else gas["alpha_a"] / (4.0 * math.pi)
    G = c["groups"]
    if G:
        for k in ("alpha_a", "alpha_s", "eta"):
            gas[k] = (gas[k][None] * uni(0.5, 2.0, G, *sh)).contiguous()
    dt = torch.float32 if c["prec"] == "f32" else torch.float64
    I = torch.zeros(((G,) if G else ()) + sh + (nap,), dtype=dt, device=DEV)
    base = (gas["T"] ** 4 / (4.0 * math.pi)).to(dt)[..., None]
    for part in (I if G else I[None]):
        part[..., :n_ang] = base * (0.9 + 0.2 * torch.rand(sh + (n_ang,), generator=g, dtype=dt, device=DEV))
    return I, {k: v.contiguous() if v is not None else None for k, v in gas.items()}


class State:
    """A problem in hand: the context and everything a step reads and writes."""

    def __init__(self, c, seed):
        self.c = c
        self.ctx = rad.rad_create(torch.cuda.current_stream())
        if c["n_zeta"]:
            self.n_ang, self.nap = rad.rad_init_angles_latlong(self.ctx, c["n_zeta"], c["n_psi"])
        else:
            self.n_ang, self.nap = rad.rad_init_angles(self.ctx, c["level"])
        xf = _faces(c)
        kind = {"cart": "mink_cart", "sph": "mink_sph", "ks": "ks_sph"}[c["metric"]]
        rad.rad_set_metric(self.ctx, kind, c["spin"], 3 if c["n3"] > 1 else 2, xf, _bc(c))
        if c["groups"]:
            rad.rad_set_groups(self.ctx, [0.25 * 2.0 ** g for g in range(c["groups"] + 1)])
        self.dt = rad.rad_cfl_dt(self.ctx, 0.3)
        self.I, self.gas = _inputs(c, seed, self.n_ang, self.nap, xf)
        self.prec = rad.RAD_F32 if c["prec"] == "f32" else rad.RAD_F64
        self.opts = rad.rad_opts_default(precision=self.prec, recon=RECON[c["recon"]],
                                         recon_ang=RECON[c["recon_ang"]], coupling=COUPLE[c["coupling"]],
                                         tau_const=c["tau"], rad_dom=int(c["rad_dom"]), gamma=GAMMA)
        sh = (c["n3"], c["n2"], c["n1"])
        G = (c["groups"],) if c["groups"] else ()
        self.src = torch.zeros(G + sh + (4,), dtype=torch.float64, device=DEV) if c["src"] else None
        self.R = torch.zeros(sh + (10,), dtype=self.I.dtype, device=DEV) if c["moments"] else None
        self.frame = FRAME[c["frame"]]
        self.method = rad.RAD_MOM_BF16X3 if c["moments"] == "bf16" else rad.RAD_MOM_SIMT
        if c["do"] == "block":
            face = (3, c["n3"], c["n2"], self.nap)
            self.send = [torch.empty(face, dtype=self.I.dtype, device=DEV) for _ in range(2)]
        if c["do"] == "grad":
            self.leaves = {"I": self.I.requires_grad_()}
            names = ["alpha_a", "alpha_s"] + (["T"] if c["coupling"] == "thermal" else ["eta"])
            for k in names:
                self.leaves[k] = self.gas[k].requires_grad_()
            self.cfg = rag.StepConfig(self.ctx, {k: self.gas[k] for k in ("rho", "u")}
                                      | {"T": self.gas["T"].detach()}, self.dt, self.opts)

    def __del__(self):
        if getattr(self, "ctx", None):
            rad.rad_destroy(self.ctx)
            self.ctx = None


def prepare(case, seed):
    return State({**DEFAULT, **case}, seed)


def run(s):
    c = s.c
    if c["do"] == "moments":
        rad.rad_moments(s.ctx, s.I, s.prec, s.frame, s.method, s.gas, s.R)
        return {"R": s.R}
    if c["do"] == "grad":
        v = s.leaves
        I, T = v["I"], v.get("T")
        for _ in range(c["steps"]):
            if T is not None:
                I, T = rag.RadStepThermalFn.apply(I, T, v["alpha_a"], v["alpha_s"], s.cfg)
            else:
                I = rag.RadStepFn.apply(I, v["alpha_a"], v["alpha_s"], v["eta"], s.cfg)
        L = rag.OuterLossFn.apply(I, s.ctx, s.prec)
        grads = torch.autograd.grad(L, list(v.values()))
        return {"L": L.detach(), **{"g_" + k: g for k, g in zip(v, grads)}}
    if c["do"] == "block":
        for stage in (1, 2):
            for side in (0, 1):
                rad.rad_halo_pack(s.ctx, s.I if stage == 1 else None, s.prec, 0, side, s.send[side])
            # the neighbour across either face is the block itself: its other face's layers
            rad.rad_step_stage(s.ctx, stage, s.I, s.gas, s.dt, s.opts, s.src,
                               {(0, 0): s.send[1], (0, 1): s.send[0]})
    else:
        rad.rad_step(s.ctx, s.I, s.gas, s.dt, s.opts, s.src)
    out = {"I": s.I, "T": s.gas["T"]}
    if s.src is not None:
        out["src"] = s.src
    if s.R is not None:
        rad.rad_moments(s.ctx, s.I, s.prec, s.frame, s.method, s.gas, s.R)
        out["R"] = s.R
    return out


# ---------------------------------------------------------------- 64-bit values

def _shift(I, d, o, bc):
    """The cell o further along x_d of every cell: periodic wrap or outflow clamp."""
    ax = 2 - d
    n = I.shape[ax]
    i = torch.arange(n, device=I.device) + o
    i = i % n if bc[d][0] == "periodic" else i.clamp(0, n - 1)
    return I.index_select(ax, i)


def _slope(x, y, z, recon):
    if recon == "dc":
        return torch.zeros_like(y)
    dl, dr = y - x, z - y
    up = dl * dr > 0.0
    return torch.where(up, dl * dr / torch.where(up, dl + dr, 1.0), 0.0)


def _root(b4, b1, b0):
    """The positive root of b4 T^4 + b1 T + b0 (b4, b1 > 0 > b0), with its derivative in the coefficients."""
    with torch.no_grad():
        T = torch.minimum(-b0 / b1, (-b0 / b4).sqrt().sqrt())
        for _ in range(60):
            T = T - (b4 * T ** 4 + b1 * T + b0) / (4.0 * b4 * T ** 3 + b1)
    return T - (b4 * T ** 4 + b1 * T + b0) / (4.0 * b4 * T ** 3 + b1).detach()


def _flat_step(c, I, T0, gas, dirs, dOm, dx, dt, bc):
    """One RK2 step in Cartesian flat space: I [n3, n2, n1, bins]."""
    four_pi = 4.0 * math.pi
    ndim = 3 if c["n3"] > 1 else 2
    nx = [dirs[:, d] for d in range(3)]
    U0 = (1.0 + gas["u"].square().sum(-1)).sqrt()

    def stage(I, I0, Tm, second):
        div = torch.zeros_like(I)
        for d in range(ndim):
            q = _slope(_shift(I, d, -1, bc), I, _shift(I, d, 1, bc), c["recon"])
            # state at a cell's upper face from below, at its lower face from above
            hi, lo = I + q, I - q
            if bc[d][0] == "outflow":
                # ghosts beyond an outflow face repeat the edge cell: zero slope there
                pos, neg = _shift(hi, d, -1, bc), _shift(lo, d, 1, bc)
                ax, n = 2 - d, I.shape[2 - d]
                pos = torch.cat([I.narrow(ax, 0, 1), pos.narrow(ax, 1, n - 1)], ax)
                neg = torch.cat([neg.narrow(ax, 0, n - 1), I.narrow(ax, n - 1, 1)], ax)
            else:
                pos, neg = _shift(hi, d, -1, bc), _shift(lo, d, 1, bc)
            div = div + nx[d] / dx[d] * torch.where(nx[d] > 0.0, hi - pos, neg - lo)
        Is = 0.5 * (I0 + I - dt * div) if second else I - dt * div
        if c["coupling"] == "none":
            return Is, Tm, torch.zeros(T0.shape + (4,), dtype=I.dtype, device=I.device)
        h = 0.5 * dt if second else dt
        nb = U0[..., None] - (gas["u"][..., None, :] * dirs).sum(-1)
        aa, als = gas["alpha_a"], gas["alpha_s"]
        den = 1.0 + nb * (aa + als)[..., None] * h
        w = Is * nb * nb * dOm
        D, Em = ((1.0 / den - 1.0) * w).sum(-1), w.sum(-1)
        A2 = h / four_pi * (dOm / (nb * den)).sum(-1)
        if c["coupling"] == "thermal":
            cv = gas["rho"] / (GAMMA - 1.0)
            b1 = cv * (1.0 - A2 * als)
            Tp = _root(A2 * aa, b1, D + A2 * als * Em - b1 * Tm)
            S = aa * Tp ** 4 + als * (Em - cv * (Tp - Tm))
        else:
            Tp = Tm
            S = four_pi * gas["eta"] + als * (D + Em + four_pi * A2 * gas["eta"]) / (1.0 - A2 * als)
        out = Is / den + h / four_pi / (den * nb ** 3) * S[..., None]
        d = (out - Is) * dOm
        x = torch.stack([-d.sum(-1)] + [(d * nx[k]).sum(-1) for k in range(3)], -1)     # change of R^0_mu
        return out, Tp, x

    I1, T1, x1 = stage(I, I, T0, False)
    I2, T2, x2 = stage(I1, I, 0.5 * (T0 + T1), True)
    return I2, T2, -(0.5 * x1 + x2)


def _flat_moments(I, u, dirs, dOm, frame):
    n4 = torch.cat([torch.ones_like(dirs[:, :1]), dirs], 1)
    pairs = [(a, b) for a in range(4) for b in range(a, 4)]
    W = torch.stack([n4[:, a] * n4[:, b] * dOm for a, b in pairs], 1)
    R = I @ W
    if frame != "fluid":
        return R
    M = torch.empty(R.shape[:-1] + (4, 4), dtype=R.dtype, device=R.device)
    for p, (a, b) in enumerate(pairs):
        M[..., a, b] = M[..., b, a] = R[..., p]
    u0 = (1.0 + u.square().sum(-1)).sqrt()
    L = torch.zeros_like(M)
    L[..., 0, 0] = u0
    for a in range(3):
        L[..., 0, a + 1] = L[..., a + 1, 0] = -u[..., a]
        for b in range(3):
            L[..., a + 1, b + 1] = u[..., a] * u[..., b] / (1.0 + u0) + (1.0 if a == b else 0.0)
    M = L @ M @ L.transpose(-1, -2)
    return torch.stack([M[..., a, b] for a, b in pairs], -1)


def exact(case, seed):
    """The flat Cartesian cases (the curved ones have no short statement of their geometry).  The angle grid's
    directions and solid angles are data of the problem, in the order that the library numbers them."""
    c = {**DEFAULT, **case}
    if c["metric"] != "cart" or c["recon"] == "ppm" or c["tau"] or c["rad_dom"] or c["groups"]:
        return None
    s = State(c, seed)
    d, w, _ = rad.rad_get_angles(s.ctx, s.n_ang)
    dirs, dOm = torch.tensor(d, device=DEV), torch.tensor(w, device=DEV)
    I = s.I.detach()[..., :s.n_ang].double()
    gas = {k: v.detach() if v is not None else None for k, v in s.gas.items()}
    bc = (("periodic", "periodic"),) * 3 if c["do"] == "block" else _bc(c)
    dx = [1.0 / n for n in (c["n1"], c["n2"], c["n3"])]
    pad = s.nap - s.n_ang
    if c["do"] == "moments":
        return {"R": _flat_moments(I, gas["u"], dirs, dOm, c["frame"])}
    if c["do"] == "grad":
        v = {"I": I.requires_grad_()}
        for k in list(s.leaves)[1:]:
            v[k] = gas[k].clone().requires_grad_()
        gas.update({k: x for k, x in v.items() if k != "I"})
        J, T = v["I"], gas["T"]
        T = v.get("T", T)
        for _ in range(c["steps"]):
            J, T, _ = _flat_step(c, J, T, gas, dirs, dOm, dx, s.dt, bc)
        L = (J[:, :, -1, :] * dOm * (dirs[:, 0] > 0.0)).sum()
        g = dict(zip(v, torch.autograd.grad(L, list(v.values()))))
        g["I"] = torch.nn.functional.pad(g["I"], (0, pad))
        return {"L": L.detach(), **{"g_" + k: x for k, x in g.items()}}
    with torch.no_grad():
        J, T, src = _flat_step(c, I, gas["T"], gas, dirs, dOm, dx, s.dt, bc)
    out = {"I": torch.nn.functional.pad(J, (0, pad)), "T": T}
    if c["src"]:
        out["src"] = src
    if c["moments"]:
        out["R"] = _flat_moments(J, gas["u"], dirs, dOm, c["frame"])
    return out
