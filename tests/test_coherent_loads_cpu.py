"""No kernel reads a state through the non-coherent load path.

``__ldg`` (``ld.global.nc``) may only read data that nothing writes while the kernel runs.
The batched kernel runs both stages in one launch, so its stage 2 reads what other CTAs
wrote in the same launch; and the stage kernels are programmatic dependents, running already
when the kernel before them still writes their input.  The grid barrier and
``griddepcontrol.wait`` order ordinary loads only.  Checked on the sources: the path is left
to the constant table of the FP64 power, and no pointer of a kernel that is launched as a
dependent or cooperatively promises the compiler (``__restrict__``) that its data is constant.
"""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1305_5536_gb300", "csrc")
STATE_KERNELS = ["dg_stage2d.cuh", "dg_stage2d_tma.cuh", "dg_stage3d.cuh", "dg_stage3m.cuh",
                 "dg_mh2d.cuh", "dg_mh3d.cuh", "dg_mh3m.cuh", "dg_batch.cu"]


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))))
def test_non_coherent_loads_read_constant_tables_only(name):
    code = _code(name)
    assert "ld.global.nc" not in code
    for arg in re.findall(r"__ldg\(([^;]*)", code):
        assert arg.startswith("&kExp2Tab["), arg


@pytest.mark.parametrize("name", STATE_KERNELS)
def test_no_constant_promise_in_kernels_that_overlap_their_input(name):
    assert "__restrict__" not in _code(name)
