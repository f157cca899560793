"""A context bound to a non-blocking stream while the legacy default stream is busy: its
tables, accumulators and control blocks are in place before its first kernels run."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1305_5536_gb300 import dg, ics

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("problems", [1, 3])
def test_context_on_its_own_stream_beside_a_busy_legacy_stream(problems):
    sizes = [(24 + 8 * i, 20) for i in range(problems)]
    us = [ics.orszag_tang(n) for n in sizes]
    flat = torch.from_numpy(np.concatenate([u.ravel() for u in us])).cuda()
    a = torch.randn(4096, 4096, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(20):
        a = torch.tanh(a @ a)  # tens of milliseconds on the default stream
    s = dg.DGSolver(configs=[dg.make_config("mhd", 2, n, precision="fp64") for n in sizes],
                    stream=side.cuda_stream)
    s.set_state(flat)
    _, dts = s.times()
    for u, n, dt in zip(us, sizes, dts):
        ref = O.Problem(O.MHD, 2, n).cfl_dt(u)[0]
        assert abs(dt - ref) < 1e-13 * ref
    s.step(1, sync=True)
    got = s.get_state()
    o = 0
    for u, n in zip(us, sizes):
        ref, flag = O.Problem(O.MHD, 2, n).run(u, 1)[::2]
        g = got[o:o + u.size] if problems > 1 else got.ravel()
        o += u.size
        assert np.abs(g - np.asarray(ref).ravel()).max() < 1e-11 * np.abs(ref).max()
    torch.cuda.synchronize()
