"""rad_step_adjoint where its kernels split the work: inner cells against cells
next to a boundary (lines of the shortest lengths with and without inner cells,
outflow and periodic, along each dimension) and chunks of x3 cells (one cell,
whole and broken groups of four, a short last chunk), against the oracle's
reverse mode.  FP64 1e-11 relative per output as the other one-step tests
(2e-10 for the thermal dL/dalpha_s, whose terms cancel), FP32 2e-4."""
import numpy as np
import pytest
import torch

import paper_2302_04283_gb300 as rad
import workloads as W
from oracle import adjoint as OA
from oracle import cfl as OCFL
from oracle import step as OS
from tests.harness import GpuCase, match_bins, oracle_gas, oracle_setup, rel_err

pytestmark = pytest.mark.gpu

OUT = ("outflow", "outflow")
PER = ("periodic", "periodic")
CASES = [
    # name, sizes, level, boundary kinds (None: the workload's), recon, coupling, precision
    ("turb3d", (5, 4, 6), 1, (PER, PER, PER), "plm", "emissivity", "f64"),
    ("turb3d", (5, 6, 5), 1, (OUT, PER, OUT), "plm", "emissivity", "f64"),
    ("turb3d", (6, 5, 7), 2, (OUT, OUT, PER), "dc", "thermal", "f64"),
    ("turb3d", (5, 5, 33), 1, (PER, OUT, OUT), "plm", "thermal", "f64"),
    ("turb3d", (5, 5, 35), 2, (PER, PER, PER), "plm", "emissivity", "f32"),
    ("turb3d", (5, 5, 42), 1, (PER, PER, PER), "plm", "thermal", "f32"),
    ("adjoint2d", (9, 7, 1), 3, None, "plm", "emissivity", "f64"),
    ("adjoint2d", (5, 5, 1), 2, None, "plm", "thermal", "f64"),
    ("torus3d_big", (6, 6, 10), 1, None, "plm", "thermal", "f64"),
    ("torus3d_big", (6, 6, 10), 2, None, "plm", "emissivity", "f32"),
]


@pytest.mark.parametrize("name,n,level,bc,recon,coupling,prec", CASES)
def test_adjoint_edges_match_oracle(name, n, level, bc, recon, coupling, prec):
    w = W.make(name, n=n, level=level)
    rng = np.random.default_rng(31)
    if bc is not None:
        w["bc"] = bc
        w["name"] += "_" + "".join(b[0][0] for b in bc)     # the oracle set-up is cached by name
    w["mode"], w["eta"] = coupling, None
    if coupling == "emissivity":
        w["eta"] = 10.0 ** rng.uniform(-1, 1, w["T"].shape) / (4 * np.pi)
    st = oracle_setup(w)
    gc = GpuCase(w)
    try:
        gmap = match_bins(gc.dir, st.ang.dir.numpy())
        dt = OCFL.cfl_dt(st, w["cfl"])
        lam = rng.normal(size=w["I0"].shape)
        lamT = rng.normal(size=w["T"].shape) if coupling == "thermal" else None
        lam_o, lamT_o, ga_o, gs_o, ge_o = OA.step_vjp(
            torch.tensor(w["I0"]), torch.tensor(w["T"]), oracle_gas(w), dt, st, OS.Opts(recon=recon, mode=coupling),
            torch.tensor(lam), None if lamT is None else torch.tensor(lamT))
        f64 = prec == "f64"
        tdt = torch.float64 if f64 else torch.float32
        o = rad.rad_opts_default(
            precision=rad.RAD_F64 if f64 else rad.RAD_F32,
            coupling=rad.RAD_COUPLE_THERMAL if coupling == "thermal" else rad.RAD_COUPLE_EMISSIVITY,
            recon=rad.RAD_RECON_PLM if recon == "plm" else rad.RAD_RECON_DC)
        Ig, lg = gc.to_gpu_I(w["I0"], gmap, tdt), gc.to_gpu_I(lam, gmap, tdt)
        ln = torch.full_like(Ig, float("nan"))
        gas = gc.gas(w)
        ga, gs, ge, lTn = (torch.zeros_like(gas["rho"]) for _ in range(4))
        lT = None if lamT is None else torch.tensor(lamT, device="cuda")
        rad.rad_step_adjoint(gc.ctx, Ig, gas, dt, o, lg, ln, lT, lTn if lamT is not None else None, ga, gs,
                             ge if coupling == "emissivity" else None)
        rad.rad_check(gc.ctx)
        tol = 1e-11 if f64 else 2e-4
        assert torch.all(ln[..., gc.n_ang:] == 0)            # padding bins are written as zeros
        assert rel_err(gc.from_gpu_I(ln, gmap), lam_o.numpy()) < tol
        assert rel_err(ga.cpu().numpy(), ga_o.numpy()) < tol
        assert rel_err(gs.cpu().numpy(), gs_o.numpy()) < (2e-10 if f64 and coupling == "thermal" else tol)
        if coupling == "emissivity":
            assert rel_err(ge.cpu().numpy(), ge_o.numpy()) < tol
        else:
            assert rel_err(lTn.cpu().numpy(), lamT_o.numpy()) < tol
    finally:
        gc.close()
