"""A batched push whose snapshots differ in size by orders of magnitude: the
slots hold what single pushes leave in them."""
import pytest
import torch

from paper_1612_07875_gb300 import sdmd as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns", [[6_000_000, 1, 5, 4096, 1000], [4097, 1], [8_388_608, 8_388_608, 17]])
def test_push_many_of_uneven_sizes(ns):
    m = 3
    hs, ref = [[S.sdmd_create(n, m, S.SDMD_F32) for n in ns] for _ in range(2)]
    try:
        for t in range(m + 1):
            g = torch.Generator(device="cuda")
            g.manual_seed(t)
            xs = [torch.randn(n, generator=g, device="cuda") for n in ns]
            S.sdmd_push_many(hs, xs)
            for h, x in zip(ref, xs):
                S.sdmd_push(h, x)
            torch.cuda.synchronize()
        G = torch.zeros((2, m, m), dtype=torch.float64, device="cuda")
        for a, b in zip(hs, ref):
            S.sdmd_rebuild(a)                  # from the slots
            S.sdmd_gram(a, G[0])
            S.sdmd_gram(b, G[1])
            assert torch.equal(G[0], G[1])
            assert S.sdmd_status(a) == S.SDMD_OK
    finally:
        for h in hs + ref:
            S.sdmd_destroy(h)
