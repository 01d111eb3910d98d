"""A keep or accept flag is set when it is not 0: masks of 255 or of mixed values update the map as
masks of 1 do."""
import numpy as np
import pytest
import torch

import oracle
import paper_2604_12942_gb300 as gs

pytestmark = pytest.mark.gpu


def T(a):
    return torch.as_tensor(a, device="cuda")


@pytest.mark.parametrize("value", [1, 2, 255, "mixed"])
@pytest.mark.parametrize("n,nn", [(1, 1), (1000, 7), (1025, 2049), (70_001, 4095)])
def test_flags_of_any_value(n, nn, value):
    rng = np.random.default_rng(n + nn)
    P = gs.n_planes(0)
    planes, m, v = (rng.normal(0, 1, (P, n)).astype(np.float32) for _ in range(3))
    new = rng.normal(0, 1, (P, nn)).astype(np.float32)
    tags, ntags = rng.integers(0, 9, n).astype(np.int32), rng.integers(9, 12, nn).astype(np.int32)

    def flags(k):
        on = rng.random(k) < 0.6
        val = rng.integers(1, 256, k) if value == "mixed" else value
        return np.where(on, val, 0).astype(np.uint8)

    keep, acc = flags(n), flags(nn)
    out = gs.map_update(T(planes), T(m), T(v), 0, T(keep), T(new), T(acc), T(tags), T(ntags))
    ref = oracle.apply_update(planes, m, v, (keep != 0).astype(np.uint8), new, (acc != 0).astype(np.uint8),
                              tags.view(np.uint32), ntags.view(np.uint32))
    for x, y in zip(out, ref):
        np.testing.assert_array_equal(x.cpu().numpy().view(y.dtype), y)
