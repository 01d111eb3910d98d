"""The backward compositing's two forms: large grids reduce two visits together, small ones and the
counted variant one at a time.  Both do the same arithmetic per visit; only the order in which the
records' totals are added differs."""
import pytest
import torch

import paper_2604_12942_gb300 as gs
import synth
from tests.gpu_helpers import gpu_forward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("size", [(2304, 2176), (2297, 2171)])
def test_large_grid_equals_one_visit_at_a_time(tile, size):
    sc = synth.uniform_box_scene(61, 3000, sh_degree=0)
    cams = [synth.camera(*size, 90.0)]
    # at least 16 (tile, region) items a resident warp, the line of the large form
    regions = -(-size[0] // tile) * -(-size[1] // tile) * (tile // 8) ** 2
    assert regions >= 16 * 32 * torch.cuda.get_device_properties(0).multi_processor_count
    out = []
    for count in (0, 1):
        ws, planes, rgb, depth, T = gpu_forward(sc, cams, gs.default_opts(tile=tile, count_fragments=count), 1 << 24)
        P = ws.layout.total_pixels
        up = torch.linspace(-1.0, 1.0, 3 * P, device="cuda")
        upd = torch.linspace(0.5, -0.5, P, device="cuda")
        grads = torch.zeros_like(planes)
        twist = torch.zeros(1, 6, device="cuda")
        ws.render_bwd(planes, 0, grads, up, upd, twist)
        torch.cuda.synchronize()
        assert ws.counters().status == 0
        out.append((grads, twist))
    (g0, t0), (g1, t1) = out
    assert float(g0.abs().max()) > 0
    # FP32 sums of the same terms in another order: up to about 1000 additions of 6e-8 each where
    # signs cancel by a factor of ten
    for a, b in zip(g0, g1):
        assert float((a - b).norm()) <= 1e-4 * float(b.norm())
    assert float((t0 - t1).norm()) <= 1e-4 * float(t1.norm())
