"""FP64 coupling with optical depths per stage up to the end of the FP64 range.
A uniform box of gas at rest, one stage: with no emission what is left of an
intensity is I / (1 + alpha dt); with thermal emission, or an emissivity of
alpha's size, the cell is in equilibrium.  1e-14 of the intensity where
nothing is left of it; else 1e-12 as the other one-step tests."""
import math

import pytest
import torch

import paper_2302_04283_gb300 as rad
import workloads as W
from tests.harness import GpuCase

pytestmark = pytest.mark.gpu

DEPTHS = [2.0 ** 880, 2.0 ** 899, 1.5 * 2.0 ** 900, 2.0 ** 980, 1.5 * 2.0 ** 1020, 1.5 * 2.0 ** 1022, 1.25 * 2.0 ** 1023]


@pytest.mark.parametrize("mode", ["absorb", "emit", "thermal"])
@pytest.mark.parametrize("depth", DEPTHS)
def test_optical_depth_to_the_end_of_the_range(depth, mode):
    w = W.make("turb3d", n=(4, 3, 3), level=2)
    gc = GpuCase(w)
    try:
        sh = (3, 3, 4)
        one = torch.ones(sh, dtype=torch.float64, device="cuda")
        dt, E0 = 1.0, 0.25                              # nothing moves in a uniform box
        I = torch.zeros(sh + (gc.n_ap,), dtype=torch.float64, device="cuda")
        I[..., :gc.n_ang] = E0 / (4.0 * math.pi)
        o = rad.rad_opts_default(coupling=rad.RAD_COUPLE_THERMAL if mode == "thermal" else rad.RAD_COUPLE_EMISSIVITY,
                                 gamma=5.0 / 3.0)
        # emissivity: source function eta / alpha = 0.5 / 4 pi
        eta = one * (depth / (8.0 * math.pi) if mode == "emit" else 0.0)
        gas = {"rho": one, "u": torch.zeros(sh + (3,), dtype=torch.float64, device="cuda"),
               "alpha_a": one * (depth / dt), "alpha_s": one * 0.0, "eta": eta, "T": one.clone()}
        rad.rad_step_stage(gc.ctx, 1, I, gas, dt, o)
        out = torch.empty((3, 3, 3, gc.n_ap), dtype=torch.float64, device="cuda")
        rad.rad_halo_pack(gc.ctx, None, rad.RAD_F64, 0, 0, out)
        rad.rad_check(gc.ctx)
        if mode == "absorb":
            E = 0.0
        elif mode == "emit":
            E = 0.5
        else:
            T = 1.0                                     # T^4 + 1.5 T = E0 + 1.5
            for _ in range(60):
                T -= (T ** 4 + 1.5 * T - E0 - 1.5) / (4.0 * T ** 3 + 1.5)
            E = T ** 4
        tol = 1e-14 * E0 if mode == "absorb" else 1e-12 * E
        assert float((out[..., :gc.n_ang] * (4.0 * math.pi) - E).abs().max()) <= tol
    finally:
        gc.close()
