"""Pair counts past 2^32: entries that each cover every tile of the largest view.  The count is
exact and the capacity error is set, whatever the count is modulo 2^32."""
import numpy as np
import pytest
import torch

import paper_2604_12942_gb300 as gs
import synth
from tests.gpu_helpers import set_vis_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1023, 1024, 1025, 2048, 2100])
def test_pairs_of_entries_covering_the_largest_view(n):
    cams = [synth.camera(16384, 16384, 9000.0)]
    ws = gs.Workspace(n, cams, gs.default_opts(tile=8), 1 << 20)
    tiles = 2048 * 2048
    assert ws.layout.total_tiles == tiles
    rec = np.zeros((n, 12), np.float32)
    rec[:, 0:2] = 8192.0
    rec[:, 2] = np.linspace(1.0, 2.0, n)
    rec[:, 7] = rec[:, 11] = np.full(n, 20_000, np.int32).view(np.float32)
    ws.region("proj", torch.float32, 12 * n).copy_(torch.as_tensor(rec.reshape(-1)))
    set_vis_bits(ws, np.ones((1, n), bool))
    ws.region("counters", torch.int32, 8).zero_()
    ws.bin_sort()
    c = ws.counters()
    assert c.status == 3 and c.n_entries == n and c.n_pairs == n * tiles
