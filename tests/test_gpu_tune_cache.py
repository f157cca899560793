"""Tile choices saved by a library with other tile shapes are tuned anew, not read as the
tiles that have their numbers now; the file's other lines stay."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
_RUN = """
import sys; sys.path.insert(0, %r)
from paper_1305_5536_gb300 import dg, ics
s = dg.DGSolver("euler", 3, (24, 20, 16), precision="fp64")
s.set_state(ics.kh3d((24, 20, 16)))
print(s.kernel_name())
""" % ROOT


def test_a_file_of_the_first_tile_set(tmp_path):
    cache = tmp_path / "cache.txt"
    old = ["eq0_d3_fp64_lim1_24x20x16_np1 1", "eq0_d2_fp64_lim1_512x512x1_np1 2"]
    cache.write_text("\n".join(old) + "\n")
    env = dict(os.environ, DG_TUNE_CACHE=str(cache))
    env.pop("DG_TILE_VARIANT", None)
    names = [subprocess.run([sys.executable, "-c", _RUN], env=env, check=True, capture_output=True,
                            text=True).stdout.strip() for _ in range(2)]
    lines = cache.read_text().split("\n")
    assert all(q in lines for q in old)
    new = [q for q in lines if "_24x20x16_np1 " in q and q not in old]
    assert len(new) == 1, lines
    # the choice made is the one the second run reads back
    tiles = ["4x4x4", "8x4x4", "8x4x2"]
    assert names[0] == names[1] and tiles[int(new[0].split()[1])] in names[0], (names, new)
