"""Split-bf16 moments with one chunk of bins per tile (64 bins or fewer) in the
fluid frame, more tiles than CTAs and a ragged last one: every tile's
velocities belong to its own cells.  Cells at rest, cells that move along one
axis and cells that move along all.  Against plain FP64 sums, 1.5e-4 of R^00
(2^-16 per product of two 8-bit halves and FP32 accumulation)."""
import numpy as np
import pytest
import torch

import paper_2302_04283_gb300 as rad

pytestmark = pytest.mark.gpu

PAIRS = [(a, b) for a in range(4) for b in range(a, 4)]


@pytest.mark.parametrize("level,latlong", [(1, None), (2, None), (None, (4, 8)), (None, (4, 16))])
@pytest.mark.parametrize("n", [(61, 37, 21), (5, 3, 2)])       # 371 tiles of 128 cells; less than one
def test_fluid_frame_of_few_bins(level, latlong, n):
    ctx = rad.rad_create(torch.cuda.current_stream())
    try:
        na, nap = rad.rad_init_angles(ctx, level) if latlong is None else rad.rad_init_angles_latlong(ctx, *latlong)
        d, w, _ = rad.rad_get_angles(ctx, na)
        rad.rad_set_metric(ctx, "mink_cart", 0.0, 3, [np.linspace(0, 1, k + 1) for k in n], (("periodic",) * 2,) * 3)
        rng = np.random.default_rng(9)
        sh = (n[2], n[1], n[0])
        I = torch.tensor(rng.uniform(0.1, 2.0, sh + (nap,)), dtype=torch.float32, device="cuda")
        u = rng.uniform(-0.4, 0.4, sh + (3,)) * (rng.uniform(size=sh + (3,)) < 0.6)
        n4 = np.concatenate([np.ones((na, 1)), d], 1)
        W = np.stack([n4[:, a] * n4[:, b] * w for a, b in PAIRS], 1)
        R = I[..., :na].double().cpu().numpy() @ W
        M, L = np.zeros(sh + (4, 4)), np.zeros(sh + (4, 4))
        for p, (a, b) in enumerate(PAIRS):
            M[..., a, b] = M[..., b, a] = R[..., p]
        u0 = np.sqrt(1 + (u * u).sum(-1))
        L[..., 0, 0] = u0
        L[..., 0, 1:] = L[..., 1:, 0] = -u
        L[..., 1:, 1:] = np.eye(3) + u[..., :, None] * u[..., None, :] / (1 + u0)[..., None, None]
        M = L @ M @ np.swapaxes(L, -1, -2)
        ref = np.stack([M[..., a, b] for a, b in PAIRS], -1)
        out = torch.full(sh + (10,), float("nan"), dtype=torch.float32, device="cuda")
        rad.rad_moments(ctx, I, rad.RAD_F32, rad.RAD_FRAME_FLUID, rad.RAD_MOM_BF16X3,
                        {"u": torch.tensor(u, device="cuda")}, out)
        rad.rad_check(ctx)
        assert (np.abs(out.double().cpu().numpy() - ref) / np.abs(ref[..., :1])).max() < 1.5e-4
    finally:
        torch.cuda.synchronize()
        rad.rad_destroy(ctx)
