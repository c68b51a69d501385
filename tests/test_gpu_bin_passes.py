"""Cell binning at the edges of its sort: bucket counts of one, two and three digits' bits (an even split of the bits over
the passes), centres below and above a tile of 2048, counts short enough for the one-block scan and too long for it.
Whole numbers: compared exactly with a stable sort on the host."""
import numpy as np
import pytest

from tests.test_gpu_cells import fga  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc", [(1, 1, 1), (1, 2, 1), (8, 8, 4), (257, 1, 1), (16, 16, 16), (41, 40, 43), (300, 1, 256)])
@pytest.mark.parametrize("n", [0, 1, 2047, 2048, 2049, 100_000, 1_500_001])
def test_bin_matches_stable_sort(fga, nc, n):  # noqa: F811
    import torch
    rng = np.random.default_rng(n + nc[0])
    Q = rng.random((n, 3)).astype(np.float32) * np.float32(1.2) - np.float32(0.1)      # some outside: clamped
    inv_h = float(max(nc))
    keys, perm, start = (t.cpu().numpy() for t in fga.bin_centres(torch.as_tensor(Q, device="cuda"), (0.0, 0.0, 0.0), inv_h, nc))
    c = np.floor((Q - np.float32(0.0)) * np.float32(inv_h)).astype(np.int64)
    c = np.minimum(np.maximum(c, 0), np.array(nc) - 1)
    want = (c[:, 0] * nc[1] + c[:, 1]) * nc[2] + c[:, 2]
    assert np.array_equal(keys[:n], want)
    assert np.array_equal(perm[:n], np.argsort(want, kind="stable"))
    assert np.array_equal(start, np.searchsorted(np.sort(want), np.arange(int(np.prod(nc)) + 1), side="left"))
