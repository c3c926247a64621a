"""bench.py's count of the reduction's launches, on the CPU: by the tiles of the
largest instance, not by its nodes."""
import bench
from paper_2508_16997_gb300 import workloads as wl


def test_reduction_launches_follow_the_tiles():
    # 32 x 3 tiles: 7 x 73 = 511, 7 x 74 = 518 (ragged: 221^2 has fewer than 512 * 96 nodes)
    assert bench.reduction_launches([wl.frm(219)]) == 1
    assert bench.reduction_launches([wl.frm(221)]) == 2
    # narrow channels: 4 x 24 tiles
    assert bench.reduction_launches([wl.channel(12287, nx=4)]) == 1
    assert bench.reduction_launches([wl.channel(12288, nx=4), wl.frm(64)]) == 2
