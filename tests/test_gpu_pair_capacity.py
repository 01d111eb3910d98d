"""A workspace too small for the pairs: the error is the same whatever else the GPU runs, and the
workspace's next call starts afresh."""
import pytest
import torch

import paper_2604_12942_gb300 as gs
import synth
from tests.gpu_helpers import planes_of

pytestmark = pytest.mark.gpu


def test_capacity_error_on_several_streams_at_once():
    """Blocks of one stream's pair scan start while another's end, so some start after the last
    chunk of their own kernel has set the error."""
    n, cams = 150_000, [synth.camera(320, 240, 300.0)]
    planes = planes_of(synth.uniform_box_scene(71, n, sh_degree=0))
    o = gs.default_opts()
    full = gs.Workspace(n, cams, o, 300 * n)
    full.project(planes, 0)
    full.bin_sort()
    want = full.counters()
    assert want.status == 0 and want.n_pairs > 10_000
    streams = [torch.cuda.Stream() for _ in range(4)]
    small = [gs.Workspace(n, cams, o, 1000 * k) for k in range(4)]
    torch.cuda.synchronize()
    for _ in range(25):
        for st, ws in zip(streams, small):
            with torch.cuda.stream(st):
                ws.project(planes, 0)
                ws.bin_sort()
    torch.cuda.synchronize()
    for ws in small:
        c = ws.counters()
        assert c.status == 3 and c.n_pairs == want.n_pairs and c.n_entries == want.n_entries
    # fewer Gaussians in view of the same workspace: it works
    away = planes.clone()
    away[0:3, 5:] = -1000.0
    small[3].project(away, 0)
    small[3].bin_sort()
    c = small[3].counters()
    assert c.status == 0 and 0 <= c.n_pairs <= 3000 and c.n_entries <= 5
