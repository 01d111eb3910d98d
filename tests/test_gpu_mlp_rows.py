"""The initialiser's network at row counts around its tiles (16 rows a warp, 128 a block) and with
buffers that are only 4-byte aligned, against the oracle."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import init_model as om
from paper_2604_12942_gb300 import _native as N
from paper_2604_12942_gb300 import learned

pytestmark = pytest.mark.gpu


def _net(seed):
    Ws, bs = om.init_weights(seed)
    rng = np.random.default_rng(seed)
    bs = [0.1 * rng.normal(size=b.shape) for b in bs]
    Ws[-1] = Ws[-1] * 10
    return Ws, bs, learned.MLP(*learned.pack_params(Ws, bs))


@pytest.mark.parametrize("n", [1, 15, 16, 17, 127, 128, 129, 1000, 40_003])
def test_inference_rows(n):
    Ws, bs, mlp = _net(3)
    x = np.random.default_rng(n).normal(size=(n, 16)).astype(np.float32)
    y = mlp.infer(torch.as_tensor(x, device="cuda")).cpu().numpy()
    ref, _ = om.mlp_forward(x, Ws, bs)
    # BF16 weights and activations on both sides; an activation may round the other way (FP32
    # sums here, exact ones there): within 1e-2 of the outputs' scale, the initialiser's tolerance
    assert np.abs(y - ref).max() <= 1e-2 * np.abs(ref).max()


@pytest.mark.parametrize("n", [1, 17, 128, 300])
def test_gradients_of_a_training_step(n):
    """m after one step from zero moments is (1 - b1) times the gradient (b1 = 0: the gradient)."""
    Ws, bs, mlp = _net(4)
    rng = np.random.default_rng(n)
    x, t = rng.normal(size=(n, 16)).astype(np.float32), rng.normal(size=(n, 16)).astype(np.float32)
    loss = float(mlp.train_step(torch.as_tensor(x, device="cuda"), torch.as_tensor(t, device="cuda"), lr=1e-3, b1=0.0))
    y, cache = om.mlp_forward(x, Ws, bs)
    gW, gb = om.mlp_backward(y, t, cache, Ws)
    ref = np.concatenate([g.ravel() for g in gW] + [g.ravel() for g in gb])
    got = mlp.m.cpu().numpy()
    assert np.linalg.norm(got - ref) <= 2e-2 * np.linalg.norm(ref)
    assert abs(loss - om.mse_loss(y, t)) <= 1e-2 * om.mse_loss(y, t)
    assert float(mlp.gw.abs().max()) == 0.0 and float(mlp.gb.abs().max()) == 0.0


def test_unaligned_buffers_give_the_same_outputs():
    Ws, bs, mlp = _net(5)
    n = 200
    x = torch.randn(n, 16, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    want = mlp.infer(x)
    xs, ys = torch.empty(16 * n + 1, device="cuda"), torch.empty(16 * n + 1, device="cuda")
    wq = torch.empty(learned.N_W + 1, dtype=torch.bfloat16, device="cuda")
    xs[1:] = x.reshape(-1)
    wq[1:] = mlp.wq
    N.check(N.lib().gs_mlp_infer(C.c_void_p(wq.data_ptr() + 2), C.c_void_p(mlp.b.data_ptr()), C.c_void_p(xs.data_ptr() + 4),
                                 n, C.c_void_p(ys.data_ptr() + 4), C.c_void_p(torch.cuda.current_stream().cuda_stream)),
            "gs_mlp_infer")
    assert torch.equal(ys[1:].reshape(n, 16), want)
