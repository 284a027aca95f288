"""The bench's bytes of ch_hull's fan group: the sampled tiles and the second
level, not the survivors that the filter's pass tests."""
import os
import re

import bench

N = 10**8


def test_fan_group_bytes():
    # 24415 tiles, every 15th is sampled
    sample = 8 * 1628 * 4096
    assert bench.fan_group_bytes(N, [69, 600_000, 118_191], [69, 7_500_000, 118_191], [1, 0, 0]) == \
        2 * sample + 24 * 7_500_000 + 12 * 600_000
    assert bench.fan_group_bytes(10_000, [10_000], [10_000], [0]) == 0
    assert bench.fan_group_bytes(100_003, [2402], [2402], [0]) == 8 * 100_003
    # no set's group moves as much as reading its points
    assert bench.fan_group_bytes(N, [10**6], [10**6], [0]) < 8 * N / 10


def test_sample_is_the_librarys():
    src = open(os.path.join(bench.ROOT, "paper_2303_10581_gb300", "csrc", "fan.cuh")).read()
    assert int(re.search(r"kFanBinTiles = (\d+);", src).group(1)) == bench.FAN_BIN_TILES
    assert "s > 16 ? 16" in src
