"""rad_step_adjoint reports what the step itself reports: a source term that
overflows in the second stage only.  One bright cell, and a scattering cell
two cells on, which the light reaches in stage 2."""
import pytest
import torch

import paper_2302_04283_gb300 as rad
import workloads as W
from tests.harness import GpuCase

pytestmark = pytest.mark.gpu


# the scattering opacity times the energy density it meets (a few 1e-3 of the bright cell's) is past the type's range
@pytest.mark.parametrize("prec,bright,scat", [("f64", 1e302, 1e12), ("f32", 1e36, 1e5)])
def test_overflow_in_the_second_stage_is_reported(prec, bright, scat):
    w = W.make("turb3d", n=(9, 3, 3), level=2)
    gc = GpuCase(w)
    try:
        sh = (3, 3, 9)
        tdt = torch.float64 if prec == "f64" else torch.float32
        zero = torch.zeros(sh, dtype=torch.float64, device="cuda")
        I = torch.zeros(sh + (gc.n_ap,), dtype=tdt, device="cuda")
        I[:, :, 0, :gc.n_ang] = bright
        as_ = zero.clone()
        as_[:, :, 2] = scat
        gas = {"rho": zero + 1.0, "u": torch.zeros(sh + (3,), dtype=torch.float64, device="cuda"), "alpha_a": zero,
               "alpha_s": as_, "eta": zero, "T": zero + 1.0}
        dt = rad.rad_cfl_dt(gc.ctx, 0.3)
        o = rad.rad_opts_default(precision=rad.RAD_F64 if prec == "f64" else rad.RAD_F32,
                                 recon=rad.RAD_RECON_DC, coupling=rad.RAD_COUPLE_EMISSIVITY)
        J = I.clone()
        rad.rad_step_stage(gc.ctx, 1, J, gas, dt, o)
        rad.rad_check(gc.ctx)                                # stage 1 stays in range
        rad.rad_step_stage(gc.ctx, 2, J, gas, dt, o)
        with pytest.raises(rad.RadError) as step:
            rad.rad_check(gc.ctx)
        gr = [torch.zeros_like(zero) for _ in range(3)]
        rad.rad_step_adjoint(gc.ctx, I, gas, dt, o, torch.ones_like(I), torch.empty_like(I), None, None, *gr)
        with pytest.raises(rad.RadError) as adj:
            rad.rad_check(gc.ctx)
        assert adj.value.status == step.value.status
    finally:
        gc.close()
