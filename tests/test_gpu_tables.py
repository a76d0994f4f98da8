"""The angular-flux tables of a spherical metric are optional: a call gives
the same bits with and without them, they are bounded, a table that
does not fit the device is left out, and a call that fits without them is not
refused because of them."""
import pytest
import torch

import paper_2302_04283_gb300 as rad
import workloads as W
from tests.harness import GpuCase

pytestmark = pytest.mark.gpu

MIB = 1 << 20


def _case(name, n, level, prec, recon_ang, latlong=None):
    w = W.make(name, n=n, level=level, latlong=latlong)
    gc = GpuCase(w)
    tdt = torch.float64 if prec == "f64" else torch.float32
    I = torch.nn.functional.pad(torch.tensor(w["I0"], dtype=tdt, device="cuda"),
                                (0, gc.n_ap - gc.n_ang)).contiguous()
    o = rad.rad_opts_default(precision=rad.RAD_F64 if prec == "f64" else rad.RAD_F32, recon_ang=recon_ang,
                             coupling=rad.RAD_COUPLE_EMISSIVITY if w["eta"] is not None else
                             rad.RAD_COUPLE_THERMAL)
    return w, gc, I, gc.gas(w), rad.rad_cfl_dt(gc.ctx, w["cfl"]), o


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("name,n,level,recon_ang,latlong", [
    ("torus3d_big", (9, 7, 8), 2, rad.RAD_RECON_DC, None),       # inner and boundary cells
    ("adjoint2d", (11, 9, 1), 3, rad.RAD_RECON_DC, None),
    ("torus3d_big", (6, 6, 4), 1, rad.RAD_RECON_MAPR, None),
    ("torus3d_big", (6, 6, 4), 2, rad.RAD_RECON_PLM, (3, 6)),
])
def test_stages_and_adjoint_without_tables(name, n, level, recon_ang, latlong, prec):
    """Run once with the tables, then captured into a graph right after the
    metric is set again: a captured call builds none."""
    w, gc, I0, gas, dt, o = _case(name, n, level, prec, recon_ang, latlong)
    try:
        g = torch.Generator(device="cuda").manual_seed(3)
        lam = torch.randn(I0.shape, generator=g, dtype=torch.float64, device="cuda").to(I0.dtype)
        thermal = gas["eta"] is None
        I, T = I0.clone(), gas["T"].clone()
        src = torch.zeros(I.shape[:-1] + (4,), dtype=torch.float64, device="cuda")
        lT = torch.randn(T.shape, generator=g, dtype=torch.float64, device="cuda") if thermal else None
        ln, lTn = torch.zeros_like(I), torch.zeros_like(T)
        ga, gs, ge = (torch.zeros_like(T) for _ in range(3))
        outs = [I, T, src, ln, lTn, ga, gs, ge]

        def calls():
            I.copy_(I0)
            T.copy_(gas["T"])
            for t in outs[2:]:
                t.zero_()
            for stage in (1, 2):
                rad.rad_step_stage(gc.ctx, stage, I, {**gas, "T": T}, dt, o, src)
            rad.rad_step_adjoint(gc.ctx, I0, gas, dt, o, lam, ln, lT, lTn if thermal else None, ga, gs,
                                 None if thermal else ge)

        calls()
        torch.cuda.synchronize()
        with_tables = [t.clone() for t in outs]
        # a context on the stream that is captured; its scratch exists before the tables are dropped
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            gc.close()
            gc = GpuCase(w)
            calls()
            rad.rad_set_metric(gc.ctx, w["kind"], w["spin"], w["ndim"], w["xf"], w["bc"])
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=s):
                calls()
            for t in outs:
                t.zero_()
            graph.replay()
        s.synchronize()
        rad.rad_check(gc.ctx)
        for a, b in zip(outs, with_tables):
            assert torch.equal(a, b)
    finally:
        gc.close()


def _fill(leave):
    """Hold all device memory but `leave` bytes."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = []
    for _ in range(4):
        free = torch.cuda.mem_get_info()[0]
        if free <= leave + 2 * MIB:
            break
        hold.append(torch.empty((free - leave) // MIB * MIB, dtype=torch.uint8, device="cuda"))
    return hold


def _adjoint(gc, I, gas, dt, o):
    lam, ln = torch.ones_like(I), torch.empty_like(I)
    gr = [torch.zeros_like(gas["T"]) for _ in range(3)]
    return lambda: rad.rad_step_adjoint(gc.ctx, I, gas, dt, o, lam, ln, None, None, *gr), [ln] + gr


# 256 x 256 columns of 162 bins in FP64: 82 MiB per intensity array, the adjoint's scratch 416 MiB, the tables
# 594 (sides) + 185 (faces) MiB
BIG = ("adjoint2d", (256, 256, 1), 4, "f64", rad.RAD_RECON_DC)


def _load_kernels():
    """Kernels are loaded on their first use, which takes device memory."""
    w, gc, I, gas, dt, o = _case("adjoint2d", (8, 8, 1), 4, "f64", rad.RAD_RECON_DC)
    rad.rad_step(gc.ctx, I, gas, dt, o)
    _adjoint(gc, I, gas, dt, o)[0]()
    gc.close()


def test_a_table_that_does_not_fit_is_not_tried_again():
    """Until the metric is set again, a step after the refusal allocates nothing."""
    _load_kernels()
    w, gc, I, gas, dt, o = _case(*BIG)
    J, K = I.clone(), I.clone()
    hold = _fill(300 * MIB)
    try:
        rad.rad_step(gc.ctx, J, gas, dt, o)
        rad.rad_check(gc.ctx)
        hold.clear()
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        rad.rad_step(gc.ctx, K, gas, dt, o)
        assert torch.cuda.mem_get_info()[0] == free
        assert torch.equal(J, K)
        rad.rad_set_metric(gc.ctx, w["kind"], w["spin"], w["ndim"], w["xf"], w["bc"])
        rad.rad_step(gc.ctx, I, gas, dt, o)
        rad.rad_check(gc.ctx)
        assert torch.cuda.mem_get_info()[0] < free - 700 * MIB
        assert torch.equal(I, K)
    finally:
        hold.clear()
        torch.cuda.empty_cache()
        gc.close()


def test_adjoint_takes_its_scratch_before_the_tables():
    _load_kernels()
    w, gc, I, gas, dt, o = _case(*BIG)
    run, outs = _adjoint(gc, I, gas, dt, o)
    hold = _fill(840 * MIB)         # the side table and the scratch do not both fit
    try:
        run()
        rad.rad_check(gc.ctx)
        assert all(torch.isfinite(t).all() for t in outs)
    finally:
        hold.clear()
        torch.cuda.empty_cache()
        gc.close()


def test_tables_make_room_for_a_later_scratch():
    _load_kernels()
    w, gc, I, gas, dt, o = _case(*BIG)
    J, K = I.clone(), I.clone()
    run, outs = _adjoint(gc, I, gas, dt, o)
    rad.rad_step(gc.ctx, J, gas, dt, o)          # builds the tables
    hold = _fill(300 * MIB)                      # less than the adjoint's scratch
    try:
        run()
        rad.rad_step(gc.ctx, K, gas, dt, o)
        rad.rad_check(gc.ctx)
        assert torch.equal(J, K)
    finally:
        hold.clear()
        torch.cuda.empty_cache()
        gc.close()


def test_a_captured_step_keeps_its_tables():
    """Tables that a captured graph reads are not given up: the graph replays
    after a call that did not fit."""
    _load_kernels()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        w, gc, I, gas, dt, o = _case(*BIG)
        J = I.clone()
        run, outs = _adjoint(gc, I, gas, dt, o)
        rad.rad_step(gc.ctx, J, gas, dt, o)
        ref = J.clone()
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            rad.rad_step(gc.ctx, J, gas, dt, o)
    hold = _fill(300 * MIB)
    try:
        with torch.cuda.stream(s):
            with pytest.raises(rad.RadError):
                run()
            J.copy_(I)
            graph.replay()
            s.synchronize()
            rad.rad_check(gc.ctx)
            assert torch.equal(J, ref)
    finally:
        hold.clear()
        torch.cuda.empty_cache()
        gc.close()


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
