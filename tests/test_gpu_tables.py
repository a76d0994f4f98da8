"""The angular-flux tables of a spherical metric are optional: they are bounded."""
import pytest
import torch

import paper_2302_04283_gb300 as rad
import workloads as W
from tests.harness import GpuCase

pytestmark = pytest.mark.gpu

MIB = 1 << 20


def test_tables_stay_within_their_bound():
    """Side and face tables and their flags count together: 4 GiB."""
    w = W.make("adjoint2d", n=(338, 338, 1), level=8, with_intensity=False)
    gc = GpuCase(w)
    try:
        gas = gc.gas(w)
        dt = rad.rad_cfl_dt(gc.ctx, w["cfl"])
        I = torch.ones((1, 338, 338, gc.n_ap), dtype=torch.float64, device="cuda")
        nbytes = I.numel() * 8 + I[..., 0].numel() * 8                # the step's scratch
        assert I.numel() * 7 * 8 < 4 << 30                            # the side table alone fits
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        rad.rad_step(gc.ctx, I, gas, dt, rad.rad_opts_default(coupling=rad.RAD_COUPLE_EMISSIVITY))
        rad.rad_check(gc.ctx)
        assert free - torch.cuda.mem_get_info()[0] <= nbytes + (4 << 30) + 64 * MIB
    finally:
        gc.close()
