"""One FP64 stage with optical depths up to the end of the FP64 range, a uniform
box of gas at rest without emission: what is left of an intensity is
I / (1 + alpha dt).  Where 1 / (1 + alpha dt) is below the normal range it counts
as zero, and so does the intensity."""
import math

import pytest
import torch

import paper_2302_04283_gb300 as rad
import workloads as W
from tests.harness import GpuCase

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth", [2.0 ** 900, 1.5 * 2.0 ** 1020, 1.5 * 2.0 ** 1022, 1.25 * 2.0 ** 1023])
def test_optical_depth_at_the_end_of_the_range(depth):
    w = W.make("turb3d", n=(4, 3, 3), level=2)
    gc = GpuCase(w)
    try:
        sh = (3, 3, 4)
        one = torch.ones(sh, dtype=torch.float64, device="cuda")
        dt = 1.0             # nothing moves in a uniform box
        I = torch.zeros(sh + (gc.n_ap,), dtype=torch.float64, device="cuda")
        I[..., :gc.n_ang] = 0.25 / (4.0 * math.pi)
        o = rad.rad_opts_default(coupling=rad.RAD_COUPLE_EMISSIVITY)
        gas = {"rho": one, "u": torch.zeros(sh + (3,), dtype=torch.float64, device="cuda"),
               "alpha_a": one * (depth / dt), "alpha_s": one * 0.0, "eta": one * 0.0, "T": one.clone()}
        rad.rad_step_stage(gc.ctx, 1, I, gas, dt, o)
        out = torch.empty((3, 3, 3, gc.n_ap), dtype=torch.float64, device="cuda")
        rad.rad_halo_pack(gc.ctx, None, rad.RAD_F64, 0, 0, out)
        rad.rad_check(gc.ctx)
        ref = 0.25 / (4.0 * math.pi) / depth if depth < 2.0 ** 1021 else 0.0
        assert float((out[..., :gc.n_ang] - ref).abs().max()) <= 1e-14 * ref
    finally:
        gc.close()
