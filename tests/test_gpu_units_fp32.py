"""FP32 in unit systems whose products leave the FP32 range although density, pressure and
velocities do not: one step against the oracle at the FP32 bar (1e-5 of each variable's
scale), and the adjoint step against the FP64 one."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1305_5536_gb300 import dg

pytestmark = pytest.mark.gpu

N = (19, 11)


def _state(gamma, rho0, c0, jump, mach, mhd=False):
    """Random cells around density rho0 and sound speed c0 (MHD: and Alfven speed c0)."""
    rng = np.random.default_rng(7)
    sh = (N[1], N[0])
    rho, p = (a * np.exp(jump * rng.uniform(-1, 1, sh)) for a in (rho0, rho0 * c0 * c0))
    c = np.sqrt(gamma * p / rho)
    vx, vy = (mach * c * rng.uniform(-1, 1, sh) for _ in range(2))
    u = np.zeros((17 if mhd else 12,) + sh)
    u[0], u[3], u[6] = rho, rho * vx, rho * vy
    u[9] = p / (gamma - 1) + 0.5 * rho * (vx ** 2 + vy ** 2)
    if mhd:
        u[12:14] = np.sqrt(rho0) * c0 * rng.uniform(-1, 1, (2,) + sh)
        u[9] += 0.5 * (u[12] ** 2 + u[13] ** 2)
    return u


def _one_step(u, gamma, integrator, limiter, mhd=False):
    P = O.Problem(O.MHD if mhd else O.EULER, 2, N, gamma=gamma, limiter=limiter)
    dt = 0.2 * P.cfl_dt(u)[0]
    ref, flag = P.mh_step(u, dt) if integrator == "mh" else P.step(u, dt)
    assert flag == 0
    s = dg.DGSolver("mhd" if mhd else "euler", 2, N, gamma=gamma, limiter=limiter, precision="fp32",
                    integrator=integrator)
    s.set_state(u)
    assert abs(s.times()[1][0] - 5 * dt) < 1e-5 * 5 * dt
    s.step(1, dt=dt, sync=True)
    d = np.abs(s.get_state() - ref)
    scale = [np.abs(u[0]).max(), 0, 0, np.abs(u[9]).max()]
    scale[1] = scale[2] = np.sqrt(scale[0] * scale[3])
    h = [0.5 / N[0], 0.5 / N[1]]
    for v in range(4):
        assert (d[3 * v] + d[3 * v + 1] * h[0] + d[3 * v + 2] * h[1]).max() < 1e-5 * scale[v], v
    if mhd:
        b = d[12] + d[16] * h[0] + d[14] * h[1], d[13] + d[15] * h[0] + d[16] * h[1]
        assert max(q.max() for q in b) < 1e-5 * np.sqrt(scale[3])


@pytest.mark.parametrize("gamma", [5.0 / 3.0, 1.4])
@pytest.mark.parametrize("integrator,limiter,jump,mach", [
    ("mh", 0, 1e-3, 1e-3), ("mh", 0, 0.3, 0.5), ("mh", 0, 2.0, 1.5), ("rk2", 1, 0.3, 0.5),
    ("rk2", 1, 2.0, 1.5), ("rk2", 2, 1e-3, 1e-3), ("rk2", 2, 0.3, 0.5)])
@pytest.mark.parametrize("rho0,c0", [(1e-20, 1.0), (1e-26, 1e6), (1e-30, 1e10), (1.0, 1.0), (1e20, 1.0)])
def test_euler_step(rho0, c0, jump, mach, integrator, limiter, gamma):
    """Density times pressure (the shock branch of the exact solver) from 1e-40 to 1e40."""
    _one_step(_state(gamma, rho0, c0, jump, mach), gamma, integrator, limiter)


@pytest.mark.parametrize("gamma", [5.0 / 3.0, 1.4])
@pytest.mark.parametrize("integrator,limiter,jump,mach", [
    ("mh", 0, 1e-3, 1e-3), ("mh", 0, 0.3, 0.5), ("rk2", 1, 0.3, 0.5)])
@pytest.mark.parametrize("rho0,c0", [
    (1.0, 1.0), (1.0, 1e-8), (1.0, 1e-9), (1.0, 2e-10),
    # rho c^3 = 1e-37: differences of energy fluxes are subnormal, and the FP32 right-hand
    # sides are widened to FP64 with subnormals flushed
    pytest.param(1e-10, 1e-9, marks=pytest.mark.xfail(reason="subnormal right-hand sides", strict=False)),
    (1.0, 1e-6), (1.0, 1e6)])
def test_mhd_step(rho0, c0, jump, mach, integrator, limiter, gamma):
    """Velocities whose fourth power (under the root of the fast speed) is subnormal in FP32,
    km/s in AU/s for one, down to where 16 of its bits are left."""
    _one_step(_state(gamma, rho0, c0, jump, mach, mhd=True), gamma, integrator, limiter, mhd=True)


@pytest.mark.parametrize("rho0,c0", [(1e-20, 1.0), (1e-26, 1e6), (1.0, 1.0), (1e20, 1.0)])
def test_euler_adjoint_step(rho0, c0):
    gamma = 1.4
    u = _state(gamma, rho0, c0, 0.3, 0.5)
    dt = 0.2 * O.Problem(O.EULER, 2, N, gamma=gamma, limiter=0).cfl_dt(u)[0]
    # adjoints of the variables in units of 1, 1/c0 and 1/c0^2: every component matters
    w = np.repeat([1.0, 1 / c0, 1 / c0, 1 / c0 ** 2], 3)[:, None, None]
    lam = torch.from_numpy(np.random.default_rng(3).normal(size=u.shape) * w).cuda()
    out = []
    for prec in ("fp64", "fp32"):
        s = dg.DGSolver("euler", 2, N, gamma=gamma, limiter=0, precision=prec)
        out.append(s.adjoint_step(lam, torch.from_numpy(u).cuda(), dt).cpu().numpy() / w)
    # 1e-4 of the adjoint's scale: the bar of the FP32 adjoint
    assert np.abs(out[1] - out[0]).max() < 1e-4 * np.abs(out[0]).max()


@pytest.mark.parametrize("gamma", [5.0 / 3.0, 1.4])
@pytest.mark.parametrize("integrator,limiter,jump,mach", [("mh", 0, 0.3, 0.5), ("rk2", 1, 0.3, 0.5)])
def test_euler_step_with_a_subnormal_square_of_the_sound_speed(jump, mach, integrator, limiter, gamma):
    _one_step(_state(gamma, 1e25, 4e-20, jump, mach), gamma, integrator, limiter)


@pytest.mark.parametrize("rho0,c0", [(1.0, 1.0), (1.0, 1e-9), (1.0, 3e-10)])
def test_mhd_adjoint_step(rho0, c0):
    """The fast speed's root and its derivative where the operand is subnormal."""
    gamma = 1.4
    u = _state(gamma, rho0, c0, 0.3, 0.5, mhd=True)
    dt = 0.2 * O.Problem(O.MHD, 2, N, gamma=gamma, limiter=0).cfl_dt(u)[0]
    w = np.concatenate([np.repeat([1.0, 1 / c0, 1 / c0, 1 / c0 ** 2], 3), np.full(5, 1 / c0)])[:, None, None]
    lam = torch.from_numpy(np.random.default_rng(3).normal(size=u.shape) * w).cuda()
    out = []
    for prec in ("fp64", "fp32"):
        s = dg.DGSolver("mhd", 2, N, gamma=gamma, limiter=0, precision=prec)
        out.append(s.adjoint_step(lam, torch.from_numpy(u).cuda(), dt).cpu().numpy() / w)
    # 1e-4 of the adjoint's scale: the bar of the FP32 adjoint
    assert np.abs(out[1] - out[0]).max() < 1e-4 * np.abs(out[0]).max()
