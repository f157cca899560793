"""Host transfers allocate nothing: the staging buffer of pageable states is part of the
context from the start, so neither the first transfer nor a later one waits for the
allocator (or stalls other contexts' work, as an allocation may)."""
import numpy as np
import pytest
import torch

from paper_1305_5536_gb300 import dg, ics

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(512, 512), (2048, 512)])  # 36 MB in one copy, 143 MB by planes
def test_pageable_transfers_do_not_allocate(n):
    u = ics.orszag_tang(n)
    warm = dg.DGSolver("mhd", 2, n, precision="fp32")  # kernels loaded, tile chosen
    warm.set_state(u)
    warm.get_state()
    s = dg.DGSolver("mhd", 2, n, precision="fp32")
    s.sync()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    s.set_state(u)
    got = s.get_state()
    assert torch.cuda.mem_get_info()[0] == free
    np.testing.assert_array_equal(got[::3][:4], u[:12:3])  # the averages come back as they went
