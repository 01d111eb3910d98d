"""The gradient of the opacity logit, o (1 - o) dL/do, where every other rounding is taken away: one
pixel at each Gaussian's mean, o = 0.75 to the bit, transmittance 1.  Of g o (1 - o) only the product
g o is then inexact."""
import numpy as np
import pytest
import torch

import paper_2604_12942_gb300 as gs
import synth
from tests.gpu_helpers import planes_of, set_vis_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [16, 8])
def test_one_rounding_of_the_logit_gradient(tile):
    grid, patch = 24, 32
    n, size = grid * grid, grid * patch
    o = gs.default_opts(tile=tile, chunk=256, alpha_max=1.0, T_min=0.0)
    cams = [synth.camera(size, size, float(size))]
    sc = synth.uniform_box_scene(41, n, sh_degree=0)
    # logits around ln 3, of which the projection turns some into 0.75 exactly
    x = np.full(n, np.log(3.0), np.float32)
    sc.opacity_logits[:] = (x.view(np.int32) + np.arange(n, dtype=np.int32) % 41 - 20).view(np.float32)
    planes = planes_of(sc)
    ws = gs.Workspace(n, cams, o, 1 << 22)
    ws.project(planes, 0)
    rec = ws.region("proj", torch.float32, 12 * n).cpu().numpy().reshape(n, 12).copy()
    hit = np.nonzero((ws.visible().cpu().numpy() != 0) & (rec[:, 3] == np.float32(0.75)))[0]
    assert hit.size > 0
    planes[10] = planes[10, int(hit[0])].clone()
    # records of our own: round Gaussians, one in the middle of each patch of pixels
    gy, gx = np.divmod(np.arange(n), grid)
    rec[:] = 0.0
    rec[:, 0], rec[:, 1] = gx * patch + patch / 2 + 0.5, gy * patch + patch / 2 + 0.5
    rec[:, 2], rec[:, 3], rec[:, 8] = 1.0, 0.75, 1.0
    rec[:, 4] = rec[:, 6] = -0.5 * np.log2(np.e) / 4.0
    rec[:, 7] = rec[:, 11] = np.full(n, 10, np.int32).view(np.float32)
    ws.region("proj", torch.float32, 12 * n).copy_(torch.as_tensor(rec.reshape(-1)))
    set_vis_bits(ws, np.ones((1, n), bool))
    ws.visible().fill_(1)
    P = size * size
    out, up = torch.zeros(4, P, device="cuda"), torch.zeros(3, size, size, device="cuda")
    g = np.random.default_rng(42).uniform(0.5, 2.0, n).astype(np.float32)
    up[0, torch.as_tensor(gy * patch + patch // 2), torch.as_tensor(gx * patch + patch // 2)] = torch.as_tensor(g, device="cuda")
    ws.bin_sort()
    ws.render_fwd(out[:3].reshape(-1), out[3])
    ws.composite_bwd(up.reshape(-1))
    grads = torch.zeros_like(planes)
    ws.project_bwd(planes, 0, grads)
    assert ws.counters().status == 0
    got, want = grads[10].cpu().numpy().astype(np.float64), g.astype(np.float64) * 0.75 * 0.25
    assert np.abs(got / want - 1.0).max() <= 2.0 ** -24
