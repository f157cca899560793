"""Rarefactions whose star pressure lies below the solver's floor, 1e-10 of the smaller
pressure, without being a vacuum: two equal states moving apart at a fraction of the
vacuum-generating speed 4 c / (gamma - 1).  The iteration rests on the floor and has
converged there; the forward step and the adjoint step are accepted as in the oracle."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1305_5536_gb300 import dg

pytestmark = pytest.mark.gpu

N = (16, 4)
STATES = [(5.0 / 3.0, 0.98), (5.0 / 3.0, 0.995), (5.0 / 3.0, 0.999), (1.4, 0.95), (1.4, 0.97),
          (1.4, 0.99), (1.1, 0.6), (1.1, 0.7), (1.1, 0.9), (1.1, 0.99)]


def _state(gamma, frac):
    """Receding halves (x < 1/2 to the left) of unit density and pressure."""
    left = np.broadcast_to(np.arange(N[0])[None, :] < N[0] // 2, (N[1], N[0]))
    v = np.where(left, -1.0, 1.0) * frac * 2 * np.sqrt(gamma) / (gamma - 1)
    u = np.zeros((12, N[1], N[0]))
    u[0], u[3], u[9] = 1.0, v, 1 / (gamma - 1) + 0.5 * v * v
    return u


@pytest.mark.parametrize("precision,bar", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("integrator", ["mh", "rk2"])
@pytest.mark.parametrize("gamma,frac", STATES)
def test_forward_step(gamma, frac, integrator, precision, bar):
    u = _state(gamma, frac)
    P = O.Problem(O.EULER, 2, N, gamma=gamma, limiter=0)
    dt = 0.02 * P.cfl_dt(u)[0]
    ref, flag = P.mh_step(u, dt) if integrator == "mh" else P.step(u, dt)
    assert flag == 0
    s = dg.DGSolver("euler", 2, N, gamma=gamma, limiter=0, precision=precision, integrator=integrator)
    s.set_state(u)
    s.step(1, dt=dt, sync=True)  # raises on any device error word
    got = s.get_state()
    scale = [np.abs(u[0]).max(), 0, 0, np.abs(u[9]).max()]
    scale[1] = scale[2] = np.sqrt(scale[0] * scale[3])
    h = [0.5 / N[0], 0.5 / N[1]]
    for v in range(4):
        d = np.abs(got[3 * v:3 * v + 3] - ref[3 * v:3 * v + 3])
        assert (d[0] + d[1] * h[0] + d[2] * h[1]).max() < bar * scale[v], v


@pytest.mark.parametrize("gamma,frac", STATES)
def test_adjoint_step(gamma, frac):
    u = torch.from_numpy(_state(gamma, frac)).cuda()
    P = O.Problem(O.EULER, 2, N, gamma=gamma, limiter=0)
    s = dg.DGSolver("euler", 2, N, gamma=gamma, limiter=0, precision="fp64", ckpt_every=1)
    lam = torch.from_numpy(np.random.default_rng(3).normal(size=(12, N[1], N[0]))).cuda()
    out = s.adjoint_step(lam, u, 0.02 * P.cfl_dt(u.cpu().numpy())[0])
    assert torch.isfinite(out).all()
