"""A step repeated on the same map: what a call accumulates into starts from zero every time."""
import pytest
import torch

import paper_2604_12942_gb300 as gs
import synth
from tests.gpu_helpers import planes_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extra", [{}, {"lambda_ssim": 0.2, "mask_erode": 2}])
@pytest.mark.parametrize("graph", [False, True])
def test_repeated_gradient_step_gives_the_same_losses_and_twists(extra, graph):
    sc = synth.uniform_box_scene(51, 4000, sh_degree=1)
    cams = [synth.camera(96, 80, 90.0), synth.camera(57, 41, 50.0, t=[0.1, 0.0, 0.2])]
    tg = synth.random_targets(52, cams)
    trgb, td = gs.pack_rgb([t["rgb"] for t in tg]), gs.pack_plane([t["depth"] for t in tg])
    step = gs.MappingStep(planes_of(sc), 1, cams, gs.default_opts(**extra))
    if graph:
        step.capture(trgb, td, optimize=False, with_twist=True)
    seen = []
    for _ in range(3):
        step.grads.zero_()
        step.replay() if graph else step(trgb, td, optimize=False, with_twist=True)
        torch.cuda.synchronize()
        assert step.ws.counters().status == 0
        seen.append((step.loss.clone(), step.twist.clone(), step.grads.clone(), step.rgb.clone()))
    for loss, twist, grads, rgb in seen[1:]:
        assert torch.equal(rgb, seen[0][3])
        # sums of float atomics: equal up to the order of the additions
        assert torch.allclose(loss, seen[0][0], rtol=1e-6)
        assert torch.allclose(twist, seen[0][1], rtol=1e-4, atol=1e-6 * float(seen[0][1].abs().max()))
        assert torch.allclose(grads, seen[0][2], rtol=1e-4, atol=1e-6 * float(seen[0][2].abs().max()))
