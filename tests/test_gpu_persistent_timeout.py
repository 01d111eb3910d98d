"""Waits of the persistent step that give up while other blocks still start or composite: the step
reports it, changes nothing, and the workspace's next step works."""
import pytest
import torch

import paper_2604_12942_gb300 as gs
import synth
from tests.gpu_helpers import planes_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("polls", [1, 4, 60])
def test_time_out_while_other_blocks_composite(polls):
    cams = [synth.camera(640, 480, 500.0)]
    tg = synth.random_targets(82, cams)
    trgb, tdep = gs.pack_rgb([t["rgb"] for t in tg]), gs.pack_plane([t["depth"] for t in tg])
    o = gs.default_opts(tile=16, chunk=256, persistent=1)
    step = gs.MappingStep(planes_of(synth.uniform_box_scene(81, 30_000, sh_degree=1)), 1, cams, o)
    before = [t.clone() for t in (step.planes, step.m, step.v)]
    for skip in (0, 1, 150) * 4:
        o.sync_skip_block, o.sync_spin_limit = skip, polls
        step(trgb, tdep)
        c = step.ws.counters()
        assert c.status == 4 and c.adam_step == 0
        for a, b in zip(before, (step.planes, step.m, step.v)):
            assert torch.equal(a, b)
    o.sync_skip_block, o.sync_spin_limit = -1, 0
    step(trgb, tdep)
    c = step.ws.counters()
    assert c.status == 0 and c.adam_step == 1
