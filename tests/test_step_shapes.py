"""Shapes the autotuner times: one per kernel that runs, and every one of them with a persistent
form where that form exists."""
import pytest
import torch

import paper_2604_12942_gb300 as gs
import synth
from paper_2604_12942_gb300 import autotune


def test_16_pixel_tiles_are_one_candidate():
    c = autotune.step_candidates()
    assert c == [(8, 32), (8, 64), (8, 128), (8, 256), (16, 256)]
    assert autotune.step_candidates(tile=16) == [(16, 256)]
    assert autotune.step_candidates(tile=8) == c[:4]
    assert autotune.step_candidates(chunk=64) == [(8, 64), (16, 64)]      # a caller's own choice stays
    assert autotune.step_candidates(16, 32) == [(16, 32)]


@pytest.mark.gpu
@pytest.mark.parametrize("chunk", [32, 64, 128, 256])
def test_persistent_step_takes_every_chunk_of_its_tile(chunk):
    from tests.gpu_helpers import planes_of
    cams = [synth.camera(160, 120, 150.0)]
    tg = synth.random_targets(92, cams)
    trgb, tdep = gs.pack_rgb([t["rgb"] for t in tg]), gs.pack_plane([t["depth"] for t in tg])
    planes = planes_of(synth.uniform_box_scene(91, 5_000, sh_degree=0))
    out = []
    for persistent in (0, 1):
        step = gs.MappingStep(planes.clone(), 0, cams, gs.default_opts(tile=16, chunk=chunk, persistent=persistent))
        loss = step(trgb, tdep).loss.clone()
        c = step.ws.counters()
        assert c.status == 0 and c.adam_step == 1
        out.append((step.rgb.clone(), loss))
    # one device function, which two kernels may contract differently: a few rounding errors a pixel
    assert torch.allclose(out[0][0], out[1][0], rtol=0, atol=1e-5)
    assert torch.allclose(out[0][1], out[1][1], rtol=1e-5)
