"""The FP64 exact Riemann solver on the GPU against the oracle, over the range of its
inputs: one MUSCL-Hancock step of piecewise constant data is one solve per face, so
weak and strong jumps, supersonic flow, near-vacuum rarefactions and unit systems
outside the FP32 range (where the FP32 first guess does not exist) reach every branch
of the first guess, the iteration and the sampling."""
import numpy as np
import pytest

import oracle as O
from paper_1305_5536_gb300 import dg

pytestmark = pytest.mark.gpu


def _state(n, gamma, jump, mach, rho0, p0, seed):
    rng = np.random.default_rng(seed)
    nx, ny = n
    rho = rho0 * np.exp(jump * rng.uniform(-1, 1, (ny, nx)))
    p = p0 * np.exp(jump * rng.uniform(-1, 1, (ny, nx)))
    c = np.sqrt(gamma * p / rho)
    vx, vy = (mach * c * rng.uniform(-1, 1, (ny, nx)) for _ in range(2))
    u = np.zeros((12, ny, nx))
    u[0], u[3], u[6] = rho, rho * vx, rho * vy
    u[9] = p / (gamma - 1) + 0.5 * rho * (vx ** 2 + vy ** 2)
    return u


@pytest.mark.parametrize("gamma", [5.0 / 3.0, 1.4, 1.1])
@pytest.mark.parametrize("jump,mach", [(0.0, 0.0), (1e-9, 1e-9), (1e-3, 1e-3), (0.3, 0.5), (2.0, 1.5),
                                       (5.0, 0.8)])
@pytest.mark.parametrize("rho0,p0", [(1.0, 1.0), (1e-24, 1e-12), (1e-60, 1e-50), (1e40, 1e50)])
def test_one_solve_per_face(gamma, jump, mach, rho0, p0):
    n = (19, 11)
    u = _state(n, gamma, jump, mach, rho0, p0, 7)
    P = O.Problem(O.EULER, 2, n, gamma=gamma, limiter=0)
    dt = 0.2 * P.cfl_dt(u)[0]
    ref, flag = P.mh_step(u, dt)
    assert flag == 0
    s = dg.DGSolver("euler", 2, n, gamma=gamma, limiter=0, precision="fp64", integrator="mh")
    s.set_state(u)
    s.step(1, dt=dt, sync=True)
    got = s.get_state()
    # 1e-12 of each variable's scale, the bar of the FP64 path (momenta: sqrt(rho E))
    scale = [np.abs(u[0]).max(), 0, 0, np.abs(u[9]).max()]
    scale[1] = scale[2] = np.sqrt(scale[0] * scale[3])
    for v in range(4):
        assert np.abs(got[3 * v] - ref[3 * v]).max() < 1e-12 * scale[v], v
        h = [0.5 / n[0], 0.5 / n[1]]
        for d in range(2):
            assert np.abs(got[3 * v + 1 + d] - ref[3 * v + 1 + d]).max() * h[d] < 1e-12 * scale[v], (v, d)
