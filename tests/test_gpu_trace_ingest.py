"""Ingest records of a batched push: the one launch that copies every stream's
snapshot is on every handle's trace, as the copies of host snapshots are."""
import numpy as np
import pytest
import torch

from paper_1612_07875_gb300 import sdmd as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("device", [True, False])
def test_push_many_records_every_handle(device):
    ns = [4096, 17, 70_000]
    hs = [S.sdmd_create(n, 3, S.SDMD_F32) for n in ns]
    try:
        S.sdmd_trace(hs[0], 1)
        S.sdmd_trace(hs[2], 1)
        for _ in range(2):
            xs = [np.ones(n, dtype=np.float32) for n in ns]
            S.sdmd_push_many(hs, [torch.from_numpy(x).cuda() for x in xs] if device else xs)
            torch.cuda.synchronize()
        assert len(S.sdmd_trace_times(hs[0], S.SDMD_K_INGEST)) == 2
        assert len(S.sdmd_trace_times(hs[1], S.SDMD_K_INGEST)) == 0     # not traced
        times = S.sdmd_trace_times(hs[2], S.SDMD_K_INGEST)
        assert len(times) == 2 and all(t > 0 for t in times)
    finally:
        for h in hs:
            S.sdmd_destroy(h)
