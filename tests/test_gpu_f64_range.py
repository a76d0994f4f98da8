"""FP64 transport slopes over a wide range of intensities: cells that differ by
up to 240 decades, equal neighbours (zero differences) and empty cells, on
flat periodic grids with sign-paired bins (level 3) and without (levels 1, 2).
Against the scheme in numpy's long double with the library's own directions
(the oracle forms an upwind flux from both of its neighbours, which is exact
only relative to the larger).  Bins with a direction component of rounding
size are left out (their upwind side is arbitrary).  Per element, relative to
the sum of the cell's and its upwind neighbours' own terms: nothing larger on
the downwind side or two cells upwind may enter.  1e-12: a few tens of
roundings of 1e-16."""
import numpy as np
import pytest
import torch

import paper_2302_04283_gb300 as rad
import workloads as W
from tests.harness import GpuCase

pytestmark = pytest.mark.gpu


def _stage(I, dirs, dx, dt, ndim, plm):
    out = I.copy()
    for d in range(ndim):
        ax = 2 - d
        lo, hi = np.roll(I, 1, ax), np.roll(I, -1, ax)
        q = np.zeros_like(I)
        if plm:
            dl, dr = I - lo, hi - I
            up = np.sign(dl) * np.sign(dr) > 0
            q[up] = dl[up] * (dr[up] / (dl[up] + dr[up]))
        n = dirs[:, d]
        fp = (I + q) - np.roll(I + q, 1, ax)            # from below
        fm = np.roll(I - q, -1, ax) - (I - q)           # from above
        out -= dt * n / dx[d] * np.where(n > 0, fp, fm)
    return out


def _scale(I, dirs, dx, dt, ndim):
    """One stage's terms without signs: the cell's and its upwind neighbours'."""
    out = I.copy()
    for d in range(ndim):
        ax, n = 2 - d, dirs[:, d]
        out += dt * np.abs(n) / dx[d] * (I + np.where(n > 0, np.roll(I, 1, ax), np.roll(I, -1, ax)))
    return out


@pytest.mark.parametrize("name,n,level,recon", [
    ("turb3d", (3, 5, 7), 3, "plm"),
    ("turb3d", (3, 6, 34), 1, "plm"),
    ("turb3d", (3, 5, 7), 1, "dc"),
    ("hotspot2d", (3, 6, 1), 2, "plm"),
])
def test_f64_slopes_over_the_range(name, n, level, recon):
    w = W.make(name, n=n, level=level)
    rng = np.random.default_rng(11)
    I = 10.0 ** rng.uniform(-120.0, 120.0, w["I0"].shape)
    I[rng.uniform(size=I.shape) < 0.15] = 0.0
    I[rng.uniform(size=I.shape[:-1]) < 0.3] = 1.0       # equal neighbours
    gc = GpuCase(w)
    try:
        Ig = torch.tensor(np.pad(I, ((0, 0),) * 3 + ((0, gc.n_ap - gc.n_ang),)), device="cuda")
        dt = rad.rad_cfl_dt(gc.ctx, 0.1)
        o = rad.rad_opts_default(coupling=rad.RAD_COUPLE_NONE,
                                 recon=rad.RAD_RECON_PLM if recon == "plm" else rad.RAD_RECON_DC)
        # one stage: its result is the context's scratch, three cells across x1
        rad.rad_step_stage(gc.ctx, 1, Ig, gc.gas(w), dt, o)
        out = torch.empty((3,) + Ig.shape[:2] + (gc.n_ap,), dtype=torch.float64, device="cuda")
        rad.rad_halo_pack(gc.ctx, None, rad.RAD_F64, 0, 0, out)
        rad.rad_check(gc.ctx)
        keep = (np.abs(gc.dir) > 1e-12).all(-1) if w["ndim"] == 3 else (np.abs(gc.dir[:, :2]) > 1e-12).all(-1)
        dirs = gc.dir[keep].astype(np.longdouble)
        J = I[..., keep].astype(np.longdouble)
        dx = [np.longdouble(x[1] - x[0]) for x in w["xf"]]
        L = np.longdouble(dt)
        ref = _stage(J, dirs, dx, L, w["ndim"], recon == "plm")
        got = out.permute(1, 2, 0, 3)[..., :gc.n_ang].cpu().numpy()[..., keep]
        assert np.all(np.abs(got - ref) <= 1e-12 * _scale(J, dirs, dx, L, w["ndim"]))
    finally:
        gc.close()
