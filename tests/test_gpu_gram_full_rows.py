"""uint8 tensor-core Gram where only some lanes of a converter warp have a row
to store (the last row group is partly filled, or holds the ones row), over
several K-steps and chunks: lanes of one warp read a staging stage that the
warp refills next, so they must not run apart. The result is whole numbers and
equals the int64 product; repeated rebuilds give the same."""
import numpy as np
import pytest
import torch

from paper_1612_07875_gb300 import sdmd as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c,k,n", [(1, 1, 5 * 1024 + 7), (3, 1, 300_001), (7, 7, 1_000_003), (8, 3, 77_824), (9, 9, 600_000),
                                   (63, 5, 200_003), (66, 66, 155_648), (127, 127, 100_001), (130, 130, 60_007),
                                   (200, 9, 40_013)])
def test_partly_filled_row_groups(c, k, n):
    rng = np.random.default_rng(c * 1000 + k)
    x = rng.integers(0, 256, (c, n), dtype=np.uint8)
    w = x.astype(np.float64)               # products below 2^16, sums below 2^53: exact
    ref = (w @ w.T).astype(np.int64)
    h = S.sdmd_create(n, c + 1, S.SDMD_U8)
    G = torch.zeros((c, c), dtype=torch.int64, device="cuda")
    try:
        for j in range(0, c - k):
            S.sdmd_push(h, torch.from_numpy(x[j]).cuda())
        S.sdmd_push_batch(h, k, torch.from_numpy(x[c - k:].copy()).cuda(), n)
        for _ in range(8):
            S.sdmd_gram(h, G)
            assert np.array_equal(G.cpu().numpy(), ref)
            S.sdmd_rebuild(h)
        assert S.sdmd_status(h) == S.SDMD_OK
    finally:
        S.sdmd_destroy(h)
