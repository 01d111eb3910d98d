"""Map-size updates at the sizes and values where their chunks, digits and cells can go wrong.
Keep and accept flags are integer decisions and the compaction copies: exact against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2604_12942_gb300 as gs

pytestmark = pytest.mark.gpu


def T(a):
    return torch.as_tensor(a, device="cuda")


@pytest.mark.parametrize("n,ratio,kind", [(1, 1.0, "normal"), (255, 0.5, "normal"), (2047, 0.1, "equal"),
                                          (2049, 0.999, "mixed"), (4097, 1.0, "mixed"), (65_537, 0.37, "equal"),
                                          (300_001, 0.01, "close"), (300_001, 0.9, "mixed")])
def test_prune_sizes(n, ratio, kind):
    rng = np.random.default_rng(n)
    lg = rng.normal(-6.0, 3.0, n).astype(np.float32)
    if kind == "equal":
        lg[:] = np.float32(-9.5)                                  # the row index alone decides
    elif kind == "close":
        lg = (np.float32(-8.0) - np.arange(n, dtype=np.float32)[::-1] * np.float32(2.0 ** -20)).astype(np.float32)
    elif kind == "mixed":
        lg[rng.random(n) < 0.1] = np.float32(-np.inf)
        lg[rng.random(n) < 0.1] = np.float32(np.nan)              # never a candidate
        lg[rng.random(n) < 0.1] = np.float32(-np.finfo(np.float32).max)
        lg[rng.random(n) < 0.1] = np.float32(np.inf)
    planes = np.zeros((gs.n_planes(0), n), np.float32)
    planes[10] = lg
    scratch = gs.map_update_scratch(n)
    pad = torch.empty(scratch.numel() + 4, dtype=torch.uint8, device="cuda")[4:]   # off every 16-byte boundary
    for s in (scratch, pad):
        keep, nk = gs.prune_plan(T(planes), 0, 0.005, ratio, s)
        ref, nk_ref = oracle.prune_plan(lg, 0.005, ratio)
        assert nk == nk_ref
        np.testing.assert_array_equal(keep.cpu().numpy(), ref)


@pytest.mark.parametrize("n,nq,radius,scale,offset", [(1, 1, 0.05, 0.04, 0.0), (3, 25, 0.05, 0.1, 0.0),
                                                      (1023, 73, 0.05, 0.3, -0.1), (1025, 24, 0.7, 2.0, 1e3),
                                                      (5000, 2000, 0.05, 0.6, 4.0e4), (5000, 2000, 0.05, 40.0, -3.0e6),
                                                      (5000, 2000, 1e-3, 100.0, 9.0e6), (3000, 2000, 30.0, 300.0, 0.0),
                                                      (2000, 500, 1e-30, 1.0, 0.0), (2000, 500, 3e38, 1e38, 0.0)])
def test_proximity_sizes_and_coordinates(n, nq, radius, scale, offset):
    """Cells from the origin to where neighbouring floats lie many cells apart, dense and sparse."""
    rng = np.random.default_rng(n + nq)
    M = (rng.uniform(-scale, scale, (3, n)) + offset * np.array([[1.0], [-1.0], [0.5]])).astype(np.float32)
    Q = (rng.uniform(-scale, scale, (3, nq)) + offset * np.array([[1.0], [-1.0], [0.5]])).astype(np.float32)
    half = nq // 2
    Q[:, :half] = M[:, rng.integers(0, n, half)]                  # at and around the radius from a map mean
    step = np.float32(radius) * rng.choice(np.float32([0, 0.5, 0.999999, 1.0, 1.000001]), half).astype(np.float32)
    with np.errstate(over="ignore"):
        Q[rng.integers(0, 3, half), np.arange(half)] += step
    for j, bad in enumerate((np.nan, np.inf, -np.inf)):
        if n > 1000:
            M[j, j] = bad
            Q[j, nq - 1 - j] = bad
    planes = np.zeros((gs.n_planes(0), n), np.float32)
    planes[0:3] = M
    with np.errstate(over="ignore", invalid="ignore"):
        ref, na_ref = oracle.dedup_plan(M, Q, radius)
    acc, na = gs.dedup_plan(T(planes), 0, T(Q), radius)
    np.testing.assert_array_equal(acc.cpu().numpy(), ref)
    assert na == na_ref


@pytest.mark.parametrize("n,nn", [(1, 0), (255, 1), (256, 256), (257, 255), (2048, 2049), (70_001, 4095)])
def test_update_sizes(n, nn):
    rng = np.random.default_rng(n)
    P = gs.n_planes(1)
    planes, m, v = (rng.normal(0, 1, (P, n)).astype(np.float32) for _ in range(3))
    keep = (rng.random(n) < 0.7).astype(np.uint8)
    buf = torch.zeros(n + 3, dtype=torch.uint8, device="cuda")[3:]   # flags off an 8-byte boundary
    buf.copy_(T(keep))
    new = rng.normal(0, 1, (P, nn)).astype(np.float32) if nn else None
    acc = (rng.random(nn) < 0.5).astype(np.uint8) if nn else None
    for a in (acc, None):
        out = gs.map_update(T(planes), T(m), T(v), 1, buf, None if new is None else T(new), None if a is None else T(a))
        ref = oracle.apply_update(planes, m, v, keep, new, a)
        for x, y in zip(out, ref):
            np.testing.assert_array_equal(x.cpu().numpy(), y)
