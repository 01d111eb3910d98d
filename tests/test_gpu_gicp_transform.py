"""The registration from transforms whose 3 x 3 part is a rotation only to FP32, or not at all: the
weights are the inverse of Sigma~_n + R Sigma~_m R^T for the R that is given."""
import numpy as np
import pytest
import torch

import paper_2604_12942_gb300 as gs
from oracle import gicp

pytestmark = pytest.mark.gpu


def _planes(rng, means):
    n = means.shape[1]
    P = np.zeros((gs.n_planes(0), n), np.float32)
    q = rng.normal(size=(4, n))
    P[0:3], P[3:6], P[6:10] = means, rng.normal(-2, 0.3, (3, n)), q / np.linalg.norm(q, axis=0)
    return P


@pytest.mark.parametrize("kind,stretch", [("fp32", 0.0), ("scaled", 1e-3), ("scaled", 0.02), ("sheared", 1e-3)])
def test_first_transform_that_is_not_quite_a_rotation(kind, stretch):
    rng = np.random.default_rng(17)
    tar = _planes(rng, rng.uniform(-5, 5, (3, 3000)) * np.array([[1.0], [1.0], [0.2]]))
    src = _planes(rng, tar[0:3, :800] + rng.normal(0, 0.02, (3, 800)))
    T0 = gicp.se3_exp([0.0, 0.0, 0.0, 0.01, 0.02, -0.01])
    if kind == "fp32":
        T0 = T0.astype(np.float32).astype(np.float64)
    elif kind == "scaled":
        T0[:3, :3] *= 1.0 + stretch
    else:
        T0[:3, :3] = T0[:3, :3] @ np.array([[1.0, stretch, 0.0], [0.0, 1.0, 0.0], [0.0, 0.0, 1.0]])
    T, res = gs.gicp_register(torch.as_tensor(src, device="cuda"), None, torch.as_tensor(tar, device="cuda"), None, 0, T0,
                              d_corr=0.5, max_iters=5)
    covs = [gicp.planar_covariance(src[6:10, m], src[3:6, m]) for m in range(src.shape[1])]
    covt = [gicp.planar_covariance(tar[6:10, m], tar[3:6, m]) for m in range(tar.shape[1])]
    T_ref, cost, cnt, it, conv = gicp.register(src[0:3], covs, tar[0:3], covt, T0, 0.5, 5, 1e-7)
    assert res.n_corr == cnt and res.iters == it
    # the same FP64 equations: the matches' FP32 coordinates are exact inputs of both sides
    np.testing.assert_allclose(T, T_ref, atol=1e-6)
    assert abs(res.cost - cost) <= 1e-5 * max(1.0, cost)
