"""sdmd_push from aligned device memory (the Gram-row kernel copies the
snapshot into its slot) against the same snapshots from host memory (copied
into the slot first): the same G, and the same slot contents as seen by
sdmd_rebuild and by later rows. Sizes: a snapshot below one 16-byte copy, tails
of n mod 16 bytes, one and several 4 KiB pieces and chunks, windows of one and
several groups of eight slots, a wrapped ring."""
import numpy as np
import pytest
import torch

from paper_1612_07875_gb300 import sdmd as S

pytestmark = pytest.mark.gpu

TYPES = {"u8": (S.SDMD_U8, torch.uint8, torch.int64), "f32": (S.SDMD_F32, torch.float32, torch.float64),
         "c64": (S.SDMD_C64, torch.complex64, torch.complex128)}


def _run(kind, frames, n, m):
    code, _, gt = TYPES[kind]
    h = S.sdmd_create(n, m, code)
    try:
        for x in frames:
            S.sdmd_push(h, x)
        S.sdmd_set_option(h, S.SDMD_OPT_REBUILD_TENSOR, 0)
        out = []
        for again in range(2):
            G = torch.zeros((m, m), dtype=gt, device="cuda")
            S.sdmd_gram(h, G)
            out.append(torch.view_as_real(G) if G.is_complex() else G)
            S.sdmd_rebuild(h)          # one row per slot, read from the ring
        assert S.sdmd_status(h) == S.SDMD_OK
        return out
    finally:
        S.sdmd_destroy(h)


@pytest.mark.parametrize("kind", ["u8", "f32", "c64"])
@pytest.mark.parametrize("n,m", [(1, 2), (3, 9), (17, 8), (1023, 24), (4097, 7), (50001, 40), (1200003, 33)])
def test_device_and_host_sources_agree(kind, n, m):
    rng = np.random.default_rng(n + m)
    count = m + 2
    if kind == "u8":
        x = rng.integers(0, 256, (count, n), dtype=np.uint8)
    else:
        x = rng.standard_normal((count, n), dtype=np.float32)
        if kind == "c64":
            x = (x + 1j * rng.standard_normal((count, n), dtype=np.float32)).astype(np.complex64)
    host = [torch.from_numpy(v.copy()) for v in x]
    dev = [v.cuda() for v in host]             # separate allocations: 16-byte aligned
    a, b = _run(kind, dev, n, m), _run(kind, host, n, m)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and torch.equal(a[0], a[1])
    if kind == "u8":
        w = x[-m:].astype(np.int64)
        assert np.array_equal(a[0].cpu().numpy(), w @ w.T)
