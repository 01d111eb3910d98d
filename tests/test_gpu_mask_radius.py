"""The interior mask at the radii and image sizes where its 64-bit rows can go wrong: the largest
disk, images narrower than a word, edges off the 32-pixel tiles; bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2604_12942_gb300 as gs
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [0, 1, 2, 7, 15, 16])
def test_mask_of_any_radius(r):
    cams = [synth.camera(w, h, 50.0) for w, h in [(33, 31), (1, 40), (200, 47), (96, 97), (17, 1)]]
    opts = gs.default_opts(mask_erode=r, mask_opacity=0.5)
    ws = gs.Workspace(1, cams, opts, 1)
    rng = np.random.default_rng(r)
    Ts = []
    for c in cams:
        T = rng.uniform(0.0, 0.49, (c["height"], c["width"])).astype(np.float32)
        T[rng.random(T.shape) < 0.002] = 0.9          # holes the disk has to find
        Ts.append(T)
    P = ws.layout.total_pixels
    ws.region("T_final", torch.float32, P).copy_(gs.pack_plane(Ts))
    callers = [(rng.random(T.shape) < 0.9).astype(np.uint8) for T in Ts]
    for caller in (None, callers):
        out = torch.full((P,), 7, dtype=torch.uint8, device="cuda")
        ws.render_mask(out, None if caller is None else gs.pack_plane(caller, dtype=torch.uint8))
        for v, M in enumerate(gs.unpack_plane(out, cams)):
            ref = oracle.render_mask(Ts[v], 0.5, r, None if caller is None else caller[v])
            np.testing.assert_array_equal(M.cpu().numpy(), ref)
