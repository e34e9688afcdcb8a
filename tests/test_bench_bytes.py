"""The bench's byte models count the launches that run: the fused launch on
every shape that has it, the tiles each path takes, and the phi^4 update's
passes."""
import re
from pathlib import Path

import bench
import paper_2302_14720_gb300 as sw

CSRC = Path(bench.__file__).parent / "paper_2302_14720_gb300" / "csrc"


def test_chain_bytes_follow_the_fused_launch():
    fused = set()
    for shape in range(sw.sw_num_shapes()):
        i = sw.sw_shape_info(shape)
        tw, th, h = i["tile_w"], i["tile_h"], i["strip_h"]
        pb = bench.phase_bytes_per_tile(tw, th)
        got = bench.chain_bytes_per_tile(tw, th, h)
        if got == pb[1] + 8 * (tw // 32) * th + pb[4]:
            fused.add(shape)
        else:
            assert got == pb[0] + pb[1] + pb[2]
    launches = (CSRC / "sw_kernels.cu").read_text()
    assert fused == {int(x) for x in re.findall(r"case (\d+): return launch_phase31_shape<", launches)}


def test_potts_tiles():
    src = (CSRC / "sw_internal.h").read_text()
    most, small, large = map(int, re.search(r"potts_shape\(int L\) { return L <= (\d+) \? (\d+) : (\d+); }", src).groups())
    for L, shape in ((most, small), (most + 1, large)):
        i = sw.sw_shape_info(shape)
        assert bench.potts_tile(L) == (i["tile_w"], i["tile_h"])


def test_phi4_bytes():
    # what the update's arrays make of each pass; the separate projection of small lattices
    assert bench.phi4_bytes_per_site(64 ** 4) == 9 + 2 + 40 + 44
    assert bench.phi4_bytes_per_site(16 ** 4) == 9 + 2 + 40 + 32 + 44
