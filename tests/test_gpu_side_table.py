"""The angular-flux prefactors read from the side table against the same step
forming them per CTA, bit for bit: rad_step builds the table of its precision
on a context's first step, rad_step_noalloc (which allocates nothing) uses one
only where it is already there.  Grids with pentagons (level 1 has only
them), hexagons and the four-sided cells of a latitude-longitude grid."""
import pytest
import torch

import paper_2302_04283_gb300 as rad
import workloads as W
from tests.harness import GpuCase

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n,level,latlong,recon_ang", [
    ((7, 6, 4), 1, None, rad.RAD_RECON_DC),
    ((7, 5, 1), 3, None, rad.RAD_RECON_DC),
    ((6, 6, 34), 2, None, rad.RAD_RECON_DC),      # more than one chunk of x3 cells
    ((6, 5, 4), 2, None, rad.RAD_RECON_MAPR),
    ((6, 5, 4), 2, (3, 6), rad.RAD_RECON_DC),
    ((6, 5, 4), 2, (5, 8), rad.RAD_RECON_PLM),
])
def test_side_table_gives_the_same_bits(n, level, latlong, recon_ang, prec):
    w = W.make("torus3d_big", n=(n[0], n[1], 4), level=level, latlong=latlong) if n[2] > 1 else \
        W.make("adjoint2d", n=n, level=level, latlong=latlong)
    if n[2] > 4:
        w = W.make("torus3d_big", n=n, level=level, latlong=latlong)
    tdt = torch.float32 if prec == "f32" else torch.float64
    out = []
    for step in (rad.rad_step_noalloc, rad.rad_step):
        gc = GpuCase(w)
        try:
            I = torch.tensor(w["I0"], dtype=tdt, device="cuda")
            I = torch.nn.functional.pad(I, (0, gc.n_ap - gc.n_ang)).contiguous()
            gas = gc.gas(w)
            src = torch.zeros(I.shape[:-1] + (4,), dtype=torch.float64, device="cuda")
            o = rad.rad_opts_default(precision=rad.RAD_F32 if prec == "f32" else rad.RAD_F64, recon_ang=recon_ang,
                                     coupling=rad.RAD_COUPLE_EMISSIVITY if w["eta"] is not None else
                                     rad.RAD_COUPLE_THERMAL)
            dt = rad.rad_cfl_dt(gc.ctx, w["cfl"])
            for _ in range(2):
                step(gc.ctx, I, gas, dt, o, src)
            rad.rad_check(gc.ctx)
            out.append((I, gas["T"], src))
        finally:
            gc.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
