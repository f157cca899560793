"""The FP64 tiles with four threads per cell (2D, both integrators) against the oracle:
grids smaller than a tile, one tile, ragged edges, several tiles, with every limiter;
and the same Courant chain as the one-thread-per-cell tiles."""
import numpy as np
import pytest

import oracle as O
from paper_1305_5536_gb300 import dg, ics

from helpers import poly_rel_err

pytestmark = pytest.mark.gpu


def _state(eq, n):
    if eq == "mhd":
        u = ics.orszag_tang(n)
        rng = np.random.default_rng(5)
        u[[0, 9]] *= 1 + 0.05 * rng.uniform(-1, 1, u[[0, 9]].shape)
        return u
    f = lambda X, Y: (1 + 0.2 * np.sin(2 * np.pi * (X + Y) + 0.31),
                      0.5 + 0.2 * np.sin(2 * np.pi * X + 0.47),
                      -0.3 + 0.2 * np.cos(2 * np.pi * Y + 0.23),
                      1 + 0.1 * np.sin(2 * np.pi * (X - 2 * Y) + 0.11))
    return ics.add_slope_noise(ics.project_2d(f, n), 0, 2, 0.05, np.random.default_rng(4))


@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("integrator,face_points,variant",
                         [("rk2", 0, 5), ("rk2", 0, 6), ("mh", 1, 3), ("mh", 1, 4), ("mh", 2, 3), ("mh", 2, 4)])
@pytest.mark.parametrize("eq", ["euler", "mhd"])
@pytest.mark.parametrize("n", [(5, 3), (8, 8), (37, 29), (64, 20)])
def test_one_and_two_steps(n, eq, integrator, face_points, variant, limiter, monkeypatch):
    monkeypatch.setenv("DG_TILE_VARIANT", str(variant))
    e = 1 if eq == "mhd" else 0
    u0 = _state(eq, n)
    P = O.Problem(e, 2, n, limiter=limiter)
    step = (lambda u, dt: P.step(u, dt)) if integrator == "rk2" else \
        (lambda u, dt: P.mh_step(u, dt, face_points=face_points))
    dt = 0.4 * P.cfl_dt(u0)[0]
    ref, f1 = step(u0, dt)
    ref2, f2 = step(ref, dt)
    s = dg.DGSolver(eq, 2, n, precision="fp64", integrator=integrator, face_points=face_points,
                    limiter=limiter)
    s.set_state(u0)
    assert "4 threads a cell" in s.kernel_name()
    if f1 == 0:
        s.step(1, dt=dt, sync=True)
        err, where = poly_rel_err(s.get_state(), ref, e, 2, P.h)
        assert err < 1e-12, (err, where)
        if f2 == 0:
            s.step(1, dt=dt, sync=True)
            err, where = poly_rel_err(s.get_state(), ref2, e, 2, P.h)
            assert err < 3e-12, (err, where)
            # the Courant step of the state reached
            assert abs(s.times()[1][0] - P.cfl_dt(ref2)[0]) < 1e-11 * P.cfl_dt(ref2)[0]
    s.close()
