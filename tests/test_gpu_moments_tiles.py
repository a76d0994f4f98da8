"""rad_moments at the edges of its tiles: one cell, tiles of 128 cells with and
without a remainder, more tiles than CTAs; bins that fill a chunk of 64, leave
a short last chunk or need many chunks; not-a-number in the padding bins, which
are not data.  Split-bf16 against plain FP64 sums at 1.5e-4 of R^00 (2^-16 per
product of two 8-bit halves and FP32 accumulation), FP64 at 1e-13 (a few tens
to hundreds of roundings of 1e-16, with some cancellation)."""
import numpy as np
import pytest
import torch

import paper_2302_04283_gb300 as rad

pytestmark = pytest.mark.gpu

PAIRS = [(a, b) for a in range(4) for b in range(a, 4)]


@pytest.mark.parametrize("n,level,latlong", [
    ((1, 1, 1), 1, None),               # 12 bins, one cell
    ((127, 1, 1), 2, None),             # 42 bins
    ((32, 4, 1), None, (4, 16)),        # 64 bins: one whole chunk, one whole tile
    ((43, 3, 1), None, (8, 16)),        # 128 bins, 129 cells
    ((31, 19, 37), 4, None),            # 162 bins: a last chunk of 34; more tiles than one per SM
    ((7, 5, 11), 5, None),              # 252 bins
    ((9, 8, 5), 8, None),               # 642 bins
    ((3, 2, 2), 11, None),              # 1212 bins: FP64 beyond its weight table
])
@pytest.mark.parametrize("frame", ["tetrad", "fluid"])
def test_moments_tiles(n, level, latlong, frame):
    ctx = rad.rad_create(torch.cuda.current_stream())
    try:
        na, nap = rad.rad_init_angles(ctx, level) if latlong is None else rad.rad_init_angles_latlong(ctx, *latlong)
        d, w, _ = rad.rad_get_angles(ctx, na)
        ndim = 1 + (n[1] > 1) + (n[2] > 1) if n[2] > 1 or n[1] > 1 else 1
        rad.rad_set_metric(ctx, "mink_cart", 0.0, ndim, [np.linspace(0, 1, k + 1) for k in n], (("periodic",) * 2,) * 3)
        rng = np.random.default_rng(5)
        sh = (n[2], n[1], n[0])
        I = np.full(sh + (nap,), np.nan)
        I[..., :na] = rng.uniform(0.1, 2.0, sh + (na,))
        u = rng.uniform(-0.4, 0.4, sh + (3,))
        n4 = np.concatenate([np.ones((na, 1)), d], 1)
        W = np.stack([n4[:, a] * n4[:, b] * w for a, b in PAIRS], 1)
        gas = {"u": torch.tensor(u, device="cuda")}
        for tdt, prec, method, tol in ((torch.float32, rad.RAD_F32, rad.RAD_MOM_BF16X3, 1.5e-4),
                                       (torch.float64, rad.RAD_F64, rad.RAD_MOM_SIMT, 1e-13)):
            Ig = torch.tensor(I, dtype=tdt, device="cuda")
            ref = Ig[..., :na].double().cpu().numpy() @ W
            if frame == "fluid":
                M = np.zeros(sh + (4, 4))
                for p, (a, b) in enumerate(PAIRS):
                    M[..., a, b] = M[..., b, a] = ref[..., p]
                u0 = np.sqrt(1 + (u * u).sum(-1))
                L = np.zeros(sh + (4, 4))
                L[..., 0, 0] = u0
                L[..., 0, 1:] = L[..., 1:, 0] = -u
                L[..., 1:, 1:] = np.eye(3) + u[..., :, None] * u[..., None, :] / (1 + u0)[..., None, None]
                M = L @ M @ np.swapaxes(L, -1, -2)
                ref = np.stack([M[..., a, b] for a, b in PAIRS], -1)
            R = torch.full(sh + (10,), float("nan"), dtype=tdt, device="cuda")
            rad.rad_moments(ctx, Ig, prec, rad.RAD_FRAME_FLUID if frame == "fluid" else rad.RAD_FRAME_TETRAD, method,
                            gas, R)
            rad.rad_check(ctx)
            err = np.abs(R.double().cpu().numpy() - ref) / np.abs(ref[..., :1])
            assert err.max() < tol
    finally:
        torch.cuda.synchronize()
        rad.rad_destroy(ctx)
