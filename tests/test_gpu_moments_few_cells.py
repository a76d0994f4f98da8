"""FP64 moments of few cells: CTAs of one to eight warps with three cells per
warp and a ragged last warp, and many bins of so few cells that each has a
warp of its own.  Against plain sums of the same 64-bit values, 1e-13 of R^00
(a few tens to hundreds of roundings of 1e-16, with some cancellation)."""
import numpy as np
import pytest
import torch

import paper_2302_04283_gb300 as rad

pytestmark = pytest.mark.gpu

PAIRS = [(a, b) for a in range(4) for b in range(a, 4)]


@pytest.mark.parametrize("n,level", [
    ((5, 1, 1), 4), ((7, 9, 11), 2), ((13, 11, 9), 3), ((17, 13, 11), 4), ((19, 17, 13), 2), ((23, 19, 16), 1),
    ((6, 6, 6), 6), ((14, 11, 8), 6),        # 362 bins: 216 cells, and one more than a wave
    ((6, 6, 6), 5), ((7, 9, 11), 3),         # 252 and 92 bins
])
@pytest.mark.parametrize("frame", [rad.RAD_FRAME_TETRAD, rad.RAD_FRAME_FLUID])
def test_moments_of_few_cells(n, level, frame):
    ctx = rad.rad_create(torch.cuda.current_stream())
    try:
        na, nap = rad.rad_init_angles(ctx, level)
        d, w, _ = rad.rad_get_angles(ctx, na)
        ndim = 3 if n[2] > 1 else 1
        rad.rad_set_metric(ctx, "mink_cart", 0.0, ndim, [np.linspace(0, 1, k + 1) for k in n], (("periodic",) * 2,) * 3)
        rng = np.random.default_rng(13)
        sh = (n[2], n[1], n[0])
        I, u = rng.uniform(0.1, 2.0, sh + (nap,)), rng.uniform(-0.4, 0.4, sh + (3,))
        n4 = np.concatenate([np.ones((na, 1)), d], 1)
        ref = I[..., :na] @ np.stack([n4[:, a] * n4[:, b] * w for a, b in PAIRS], 1)
        if frame == rad.RAD_FRAME_FLUID:
            M, L = np.zeros(sh + (4, 4)), np.zeros(sh + (4, 4))
            for p, (a, b) in enumerate(PAIRS):
                M[..., a, b] = M[..., b, a] = ref[..., p]
            u0 = np.sqrt(1 + (u * u).sum(-1))
            L[..., 0, 0] = u0
            L[..., 0, 1:] = L[..., 1:, 0] = -u
            L[..., 1:, 1:] = np.eye(3) + u[..., :, None] * u[..., None, :] / (1 + u0)[..., None, None]
            M = L @ M @ np.swapaxes(L, -1, -2)
            ref = np.stack([M[..., a, b] for a, b in PAIRS], -1)
        out = torch.full(sh + (10,), float("nan"), dtype=torch.float64, device="cuda")
        rad.rad_moments(ctx, torch.tensor(I, device="cuda"), rad.RAD_F64, frame, rad.RAD_MOM_SIMT,
                        {"u": torch.tensor(u, device="cuda")}, out)
        rad.rad_check(ctx)
        assert (np.abs(out.cpu().numpy() - ref) / np.abs(ref[..., :1])).max() < 1e-13
    finally:
        torch.cuda.synchronize()
        rad.rad_destroy(ctx)
