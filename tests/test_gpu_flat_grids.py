"""3D Euler grids of one to three planes in FP64, through every tile shape, against the
oracle (the 8x4x2 tile is the one that such grids fill)."""
import numpy as np
import pytest

import oracle as O
from paper_1305_5536_gb300 import dg, ics

from helpers import poly_rel_err

pytestmark = pytest.mark.gpu

TILES = ["4x4x4", "8x4x4", "8x4x2"]


@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("variant", range(3))
@pytest.mark.parametrize("n", [(9, 5, 1), (16, 12, 2), (19, 7, 3)])
def test_one_step(n, variant, limiter, monkeypatch):
    monkeypatch.setenv("DG_TILE_VARIANT", str(variant))
    u = ics.kh3d(n)
    rng = np.random.default_rng(6)
    u[0::4] *= 1 + 0.02 * rng.uniform(-1, 1, u[0::4].shape)
    P = O.Problem(O.EULER, 3, n, limiter=limiter)
    dt = 0.4 * P.cfl_dt(u)[0]
    ref, flag = P.step(u, dt)
    assert flag == 0
    s = dg.DGSolver("euler", 3, n, precision="fp64", limiter=limiter)
    s.set_state(u)
    assert TILES[variant] in s.kernel_name()
    s.step(1, dt=dt, sync=True)
    err, where = poly_rel_err(s.get_state(), ref, 0, 3, P.h)
    assert err < 1e-12, (err, where)
