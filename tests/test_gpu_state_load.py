"""The one-launch state load and save: every problem of a context, all planes, the
Courant step of each problem, at sizes around the blocks of the launch (one cell, a
partial block, several blocks, more cells than the grid has threads)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1305_5536_gb300 import dg

pytestmark = pytest.mark.gpu


def _state(eq, dim, n, rng):
    """Smooth-valued random averages (positive density and pressure) and random slopes."""
    nt = dim + 2
    npl = nt * (dim + 1) + ((5 if dim == 2 else 11) if eq == "mhd" else 0)
    u = rng.uniform(-0.3, 0.3, (npl,) + tuple(reversed(n)))
    u[0] = 1.0 + 0.2 * rng.uniform(-1, 1, u[0].shape)
    u[(nt - 1) * (dim + 1)] = 3.0 + 0.2 * rng.uniform(-1, 1, u[0].shape)
    return u


@pytest.mark.parametrize("where", ["device", "pageable", "pinned"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("eq,dim,sizes", [
    ("euler", 2, [(1, 1), (17, 5), (64, 48), (255, 1), (16, 16), (257, 1)]),
    ("mhd", 2, [(33, 7), (1, 1), (600, 530)]),
    ("euler", 3, [(5, 3, 7), (16, 16, 4)]),
    ("mhd", 3, [(4, 4, 4), (9, 8, 7)]),
    ("euler", 2, [(700, 560)]),
])
def test_round_trip_and_courant_step(eq, dim, sizes, precision, where):
    rng = np.random.default_rng(3)
    us = [_state(eq, dim, n, rng) for n in sizes]
    flat = np.concatenate([u.ravel() for u in us])
    s = dg.batch([dg.make_config(eq, dim, n, precision=precision) for n in sizes])
    # twice: the accumulators of the first load are clean for the second
    for k in range(2):
        if where == "pageable":
            s.set_state(flat)
            got = s.get_state(out=np.empty_like(flat))
        else:
            t = torch.from_numpy(flat)
            t = t.cuda() if where == "device" else t.pin_memory()
            o = torch.empty_like(t) if where == "device" else torch.empty_like(t).pin_memory()
            s.set_state(t)
            got = s.get_state(out=o).cpu().numpy()
        o = 0
        _, dts = s.times()
        for u, n, dt in zip(us, sizes, dts):
            g = got[o:o + u.size].reshape(u.shape)
            o += u.size
            nt = dim + 2
            avg = [v * (dim + 1) for v in range(nt)]
            if eq == "mhd":
                avg += list(range(nt * (dim + 1), nt * (dim + 1) + dim))
            for p in range(u.shape[0]):
                want = u[p] if p in avg or precision == "fp64" else u[p].astype(np.float32).astype(np.float64)
                assert np.array_equal(g[p], want), p
            P = O.Problem(O.MHD if eq == "mhd" else O.EULER, dim, n)
            ref = P.cfl_dt(u)[0]
            # a few roundings of the arithmetic type
            assert abs(dt - ref) < (1e-14 if precision == "fp64" else 2e-6) * ref
        s.sync()
