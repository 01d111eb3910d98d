"""bench.py's count of the kernels one step launches."""
import types

import pytest

import bench


@pytest.mark.parametrize("n,views,tiles,sms,launches", [
    (2_000_000, 8, 23920, 152, 22),     # the bench's workload: a count kernel before the compaction
    (10_000, 1, 300, 152, 20),          # one wave of compaction blocks, one tile-sort pass
    (10_000, 1, 1, 152, 19),            # one tile: nothing to sort by
    (1_245_184, 1, 4800, 152, 21),      # 608 blocks of 64 words: 4 on each of 152 SMs
    (1_245_185, 1, 4800, 152, 22),
    (1_245_184, 1, 4800, 148, 22)])
def test_launches_per_step(n, views, tiles, sms, launches):
    L = types.SimpleNamespace(n=n, n_views=views, total_tiles=tiles)
    assert bench.launches_per_step(L, sms) == launches
