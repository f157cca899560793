"""The shipped tile choices belong to the tile shapes that are compiled: every key carries
the number of the set (``kTileSet`` of ``csrc/dg_capi.cu``), which is raised when an index
changes its meaning, and files of another set are not read."""
import os
import re

PKG = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1305_5536_gb300")


def test_shipped_choices_are_of_the_compiled_tile_set():
    with open(os.path.join(PKG, "csrc", "dg_capi.cu")) as f:
        number = re.search(r"constexpr int kTileSet = (\d+);", f.read()).group(1)
    with open(os.path.join(PKG, "tune_cache.txt")) as f:
        entries = [line.split() for line in f if line.strip()]
    assert entries
    for key, index in entries:
        assert re.fullmatch(r"t%s_eq[01]_d[23]_fp(32|64)_lim[012]_\d+x\d+x\d+_np\d+(_mh[12])?" % number, key), key
        assert 0 <= int(index) < 7
