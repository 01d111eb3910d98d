"""The voxel fit at point counts around its chunk sizes (32 lanes, 512 stashed points, the minimum
of 5), with voxels starting anywhere among a warp's 32 sorted positions, against FP64 NumPy; and
with output buffers that are only 4-byte aligned."""
import ctypes as C

import numpy as np
import pytest
import torch

import synth
from paper_2604_12942_gb300 import _native as N
from paper_2604_12942_gb300 import learned
from paper_2604_12942_gb300.core import camera_array

pytestmark = pytest.mark.gpu

COUNTS = [1, 4, 5, 6, 31, 32, 33, 64, 255, 256, 257, 511, 512, 513, 1025, 1500]


def _points(order, seed=2):
    """One voxel (0.5 m) per count along x, points spread anisotropically inside it, shuffled."""
    rng = np.random.default_rng(seed)
    pts, vox = [], []
    for v, k in enumerate(order):
        c = np.array([0.5 * v + 0.25, 0.25, 0.25])
        pts.append(c + np.clip(rng.normal(0, [0.09, 0.05, 0.025], (k, 3)), -0.24, 0.24))
        vox += [v] * k
    p = np.concatenate(pts).astype(np.float32)
    perm = rng.permutation(len(p))
    return p[perm].T.copy(), np.asarray(vox)[perm]


@pytest.mark.parametrize("order", [COUNTS, COUNTS[::-1], [5] * 70 + [1500] + [3] * 40, [2]])
def test_statistics_of_every_count(order):
    p, vox = _points(order)
    cam = synth.camera(64, 48, 50.0)
    dev = torch.as_tensor(p, device="cuda")
    out = learned.voxel_pca(dev, torch.rand_like(dev), cam)
    x, has, s = (out[k].cpu().numpy() for k in ("x", "has_feature", "s_pca"))
    for v, k in enumerate(order):
        rows = np.nonzero(vox == v)[0]
        assert (has[rows] == (k >= 5)).all()
        if k < 5:
            assert (x[rows] == 0).all() and (s[rows] == 0).all()
            continue
        d = p[:, rows].astype(np.float64)
        lam = np.linalg.eigvalsh(np.cov(d, bias=True))
        lam = np.maximum(lam, 1e-4)
        # FP32 sums of up to 1500 points of a few cm: the initialiser's tolerance on ln lambda
        ok = lam > 2e-4
        np.testing.assert_allclose(x[rows][:, :3][:, ok], np.broadcast_to(np.log(lam), (k, 3))[:, ok], atol=2e-3)
        np.testing.assert_allclose(s[rows], 0.5 * x[rows][:, :3], rtol=1e-6)
        assert (x[rows] == x[rows[0]])[:, :12].all()      # one fit for the voxel's points


def test_unaligned_outputs_are_the_same():
    p, _ = _points(COUNTS)
    n = p.shape[1]
    cam = synth.camera(64, 48, 50.0)
    pts = torch.as_tensor(p, device="cuda")
    col = torch.rand_like(pts)
    want = learned.voxel_pca(pts, col, cam)
    out = {k: torch.zeros(v.numel() + 1, dtype=v.dtype, device="cuda") for k, v in want.items()}
    ws = torch.empty(int(N.lib().gs_pca_workspace_size(n)), dtype=torch.uint8, device="cuda")
    opts, arr = learned.pca_opts(), camera_array([cam])
    ptr = [C.c_void_p(out[k].data_ptr() + out[k].element_size())
           for k in ("x", "has_feature", "reliable", "s_pca", "q_pca", "depth", "inside")]
    N.check(N.lib().gs_voxel_pca(C.c_void_p(pts.data_ptr()), C.c_void_p(col.data_ptr()), n, arr, 1, C.byref(opts),
                                 C.c_void_p(ws.data_ptr()), ws.numel(), *ptr,
                                 C.c_void_p(torch.cuda.current_stream().cuda_stream)), "gs_voxel_pca")
    for k, v in want.items():
        assert torch.equal(out[k][1:], v.reshape(-1)), k
