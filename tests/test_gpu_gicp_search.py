"""The correspondence search of the loop registration at its edges -- one target, target counts
around the hash's bucket counts, balls of one cell to many, queries without a match beside the
targets, coordinates FP32 cannot resolve -- against the oracle's brute force."""
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


@pytest.mark.parametrize("n_tar,d_corr", [(7, 1.0), (600, 0.05), (4096, 0.3), (5000, 1.0), (5000, 4.0)])
def test_registration_with_unmatched_rows_matches_brute_force(n_tar, d_corr):
    rng = np.random.default_rng(n_tar)
    tar = _planes(rng, rng.uniform(-3, 3, (3, n_tar)) * np.array([[1.0], [1.0], [0.1]]))
    k = min(n_tar, 700)
    near = tar[0:3, :k] + rng.normal(0, 0.1 * d_corr, (3, k))
    beside = rng.uniform(-3, 3, (3, 150)) + np.array([[0.0], [0.0], [1.2 * d_corr + 0.3]])
    src = _planes(rng, np.concatenate([near, beside, rng.uniform(90, 99, (3, 50))], 1))
    S, D = torch.as_tensor(src, device="cuda"), torch.as_tensor(tar, device="cuda")
    T, res = gs.gicp_register(S, None, D, None, 0, np.eye(4), d_corr=d_corr, max_iters=3)
    covs = [gicp.planar_covariance(src[6:10, m], src[3:6, m]) for m in range(src.shape[1])]
    covt = [gicp.planar_covariance(tar[6:10, m], tar[3:6, m]) for m in range(n_tar)]
    T_ref, cost, cnt, it, conv = gicp.register(src[0:3], covs, tar[0:3], covt, np.eye(4), d_corr, 3, 1e-7)
    assert res.n_corr == cnt and res.iters == it and res.converged == int(conv)
    np.testing.assert_allclose(T, T_ref, atol=1e-6)
    assert abs(res.cost - cost) <= 1e-5 * max(1.0, cost)


@pytest.mark.parametrize("offset", [0.0, 1e5, 3e7])
@pytest.mark.parametrize("n_tar,d_corr", [(1, 1.0), (900, 1.0), (900, 1e-4), (900, float("inf"))])
def test_exact_matches_are_found_at_any_magnitude(offset, n_tar, d_corr):
    """Source rows equal to target rows match at distance 0, the others (100 m away) do not: the
    residuals are 0, the transform stays the identity."""
    rng = np.random.default_rng(3)
    tar = _planes(rng, rng.uniform(-20, 20, (3, n_tar)) + offset)
    far = np.isinf(d_corr)
    extra = np.zeros((3, 0)) if far else rng.uniform(-20, 20, (3, 40)) + offset + np.array([[100.0], [0.0], [0.0]])
    src = _planes(rng, np.concatenate([tar[0:3, ::2], extra], 1))
    T, res = gs.gicp_register(torch.as_tensor(src, device="cuda"), None, torch.as_tensor(tar, device="cuda"), None, 0,
                              np.eye(4), d_corr=d_corr, max_iters=2)
    assert res.n_corr == tar[:, ::2].shape[1]
    assert res.cost == 0.0
    np.testing.assert_array_equal(T, np.eye(4))
