"""The temperature of the thermal coupling outside the FP32 range: gas
temperatures and heat capacities whose cube, slope or product FP32 cannot
hold.  A uniform periodic box of gas at rest with isotropic intensities, where
transport does nothing and a step is a recursion of scalars, which the test
evaluates in 64 bits (gradients by torch.autograd).  FP64: 1e-12 for the
step and 1e-11 for the gradient, as the other one-step tests (some hundred
roundings of 1e-16; dL/dalpha_s 2e-10, whose terms cancel).  FP32 intensities:
the gradient 2e-4, as there."""
import math

import pytest
import torch

import paper_2302_04283_gb300 as rad
import workloads as W
from tests.harness import GpuCase

pytestmark = pytest.mark.gpu


def _root(b4, b1, b0):
    with torch.no_grad():
        T = torch.minimum(-b0 / b1, (-b0 / b4).sqrt().sqrt())
        for _ in range(80):
            T = T - (b4 * T ** 3 * T + b1 * T + b0) / (4.0 * b4 * T ** 3 + b1)
    # one step more, whose derivative in the coefficients is the root's
    return T - (b4 * T ** 3 * T + b1 * T + b0) / (4.0 * b4 * T ** 3 + b1).detach()


def _step(E, T, aa, as_, cv, a, dt):
    """E = 4 pi I and T after one RK2 step."""
    E0, T0 = E, T
    for h, second in ((dt, False), (0.5 * dt, True)):
        Es, Tm = (0.5 * (E0 + E), 0.5 * (T0 + T)) if second else (E0, T0)
        den = 1.0 + (aa + as_) * h
        A2 = h / den
        b1 = cv * (1.0 - A2 * as_)
        Tp = _root(A2 * aa * a, b1, (1.0 / den - 1.0) * Es + A2 * as_ * Es - b1 * Tm)
        S = aa * a * Tp ** 3 * Tp + as_ * (Es - cv * (Tp - Tm))
        E, T = Es / den + h * S / den, Tp
    return E, T


# gas temperature and density (a_rad follows: gas and radiation energy are of one size)
CASES = [(1.0, 1.0), (1e12, 1.0), (8e12, 1.0), (1e13, 1.0), (1e13, 1e10), (1e20, 1.0), (1e-13, 1.0),
         (1.0, 4e37), (1.0, 1e39), (1.0, 1e-38), (1.0, 1e-45)]


def _problem(T0, rho, hot, prec):
    w = W.make("turb3d", n=(4, 3, 3), level=2)
    gc = GpuCase(w)
    sh = (3, 3, 4)
    full = lambda v: torch.full(sh, v, dtype=torch.float64, device="cuda")
    dt = rad.rad_cfl_dt(gc.ctx, 0.3)
    cv, a = 1.5 * rho, rho / T0 ** 3
    E0, aa, as_ = hot * a * T0 ** 3 * T0, 1.0 / dt, 0.5 / dt
    tdt = torch.float64 if prec == "f64" else torch.float32
    I = torch.zeros(sh + (gc.n_ap,), dtype=tdt, device="cuda")
    I[..., :gc.n_ang] = E0 / (4.0 * math.pi)
    gas = {"rho": full(rho), "u": torch.zeros(sh + (3,), dtype=torch.float64, device="cuda"), "alpha_a": full(aa),
           "alpha_s": full(as_), "eta": None, "T": full(T0)}
    o = rad.rad_opts_default(precision=rad.RAD_F64 if prec == "f64" else rad.RAD_F32, a_rad=a, gamma=5.0 / 3.0)
    x = [torch.tensor(v, dtype=torch.float64, requires_grad=True) for v in (E0, T0, aa, as_)]
    return gc, I, gas, dt, o, x, (cv, a)


def _err(got, ref):
    return float((got.double().cpu() / ref - 1.0).abs().max())


@pytest.mark.parametrize("hot", [6.0, 0.2])
@pytest.mark.parametrize("T0,rho", CASES)
def test_step_finds_the_root(T0, rho, hot):
    gc, I, gas, dt, o, x, (cv, a) = _problem(T0, rho, hot, "f64")
    try:
        rad.rad_step(gc.ctx, I, gas, dt, o)
        rad.rad_check(gc.ctx)
        with torch.no_grad():
            E, T = _step(*x, cv, a, dt)
        assert _err(gas["T"], T) < 1e-12
        assert _err(I[..., :gc.n_ang] * (4.0 * math.pi), E) < 1e-12
    finally:
        gc.close()


@pytest.mark.parametrize("hot", [6.0, 0.2])
@pytest.mark.parametrize("T0,rho,prec", [c + ("f64",) for c in CASES] + [(1.0, 1.0, "f32"), (1e13, 1.0, "f32"),
                                                                          (1e20, 1.0, "f32"), (1e-13, 1.0, "f32")])
def test_gradient_at_the_root(T0, rho, hot, prec):
    """Gradient of the summed temperature after the step."""
    gc, I, gas, dt, o, x, (cv, a) = _problem(T0, rho, hot, prec)
    try:
        lam, ln = torch.zeros_like(I), torch.empty_like(I)
        lT, lTn, ga, gs = torch.ones_like(gas["T"]), *(torch.zeros_like(gas["T"]) for _ in range(3))
        rad.rad_step_adjoint(gc.ctx, I, gas, dt, o, lam, ln, lT, lTn, ga, gs)
        rad.rad_check(gc.ctx)
        gE, gT, gaa, gas_ = torch.autograd.grad(_step(*x, cv, a, dt)[1], x)
        tol = 1e-11 if prec == "f64" else 2e-4
        dOm = torch.tensor(gc.dOmega, device="cuda")
        assert _err(ln[..., :gc.n_ang].double() / dOm, gE) < tol       # E = sum of I dOmega
        assert _err(lTn, gT) < tol
        assert _err(ga, gaa) < tol
        # scattering alone moves no energy of isotropic radiation and gas at rest: the terms cancel
        assert float((gs.cpu() - gas_).abs().max() / gaa.abs()) < (2e-10 if prec == "f64" else tol)
    finally:
        gc.close()
