"""Calls with cluster launches and programmatic launches, captured into a CUDA
graph and replayed: the results of the graph are those of the direct calls."""
import numpy as np
import pytest
import torch

from paper_1612_07875_gb300 import sdmd as S

pytestmark = pytest.mark.gpu


def _u8(count, n, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randint(0, 256, (count, n), dtype=torch.uint8, device="cuda", generator=g)


def _replay(call):
    """Capture call(stream) and run the graph once."""
    st, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=st, capture_error_mode="relaxed"):
        call(st)
    graph.replay()
    torch.cuda.synchronize()
    return graph


@pytest.mark.parametrize("m,k", [(100, 8), (200, 70)])
def test_push_batch_and_rebuild(m, k):
    n = 50_003
    x = _u8(m + k, n, m)
    hs = [S.sdmd_create(n, m, S.SDMD_U8) for _ in range(2)]
    G = torch.zeros((3, m, m), dtype=torch.int64, device="cuda")
    try:
        for h in hs:
            S.sdmd_push_batch(h, m, x[:m].contiguous(), n)       # (allocates the pass's scratch)
        new = x[m:].contiguous()
        S.sdmd_push_batch(hs[0], k, new, n)
        S.sdmd_gram(hs[0], G[0])
        keep = [_replay(lambda st: (S.sdmd_push_batch(hs[1], k, new, n, st), S.sdmd_gram(hs[1], G[1], st))),
                _replay(lambda st: (S.sdmd_rebuild(hs[1], st), S.sdmd_gram(hs[1], G[2], st)))]
        w = x[k:].cpu().numpy().astype(np.float64)
        assert np.array_equal(G[0].cpu().numpy(), (w @ w.T).astype(np.int64))
        assert torch.equal(G[1], G[0]) and torch.equal(G[2], G[0])
        assert all(S.sdmd_status(h) == S.SDMD_OK for h in hs)
        del keep
    finally:
        for h in hs:
            S.sdmd_destroy(h)


@pytest.mark.parametrize("kind,m,r", [("u8", 60, 10), ("u8", 100, 10), ("u8", 200, 10), ("c64", 40, 8), ("c64", 50, 10)])
def test_modes(kind, m, r):
    n = 5000
    h = S.sdmd_create(n, m, S.SDMD_U8 if kind == "u8" else S.SDMD_C64)
    lam = torch.zeros((2, r), dtype=torch.complex128, device="cuda")
    phi = torch.zeros((2, r, n), dtype=torch.complex64, device="cuda")
    rank = torch.zeros(2, dtype=torch.int32, device="cuda")
    try:
        g = torch.Generator(device="cuda")
        g.manual_seed(m)
        for row in _u8(m, n, m):
            x = row if kind == "u8" else torch.complex(row.float(), torch.randn(n, generator=g, device="cuda"))
            S.sdmd_push(h, x)
            torch.cuda.synchronize()
        S.sdmd_modes(h, r, phi[0], lam[0], rank[:1])
        graph = _replay(lambda st: S.sdmd_modes(h, r, phi[1], lam[1], rank[1:], st))
        assert torch.equal(*torch.view_as_real(lam)) and torch.equal(*torch.view_as_real(phi))
        assert int(rank[0]) == int(rank[1]) == r
        del graph
    finally:
        S.sdmd_destroy(h)


def test_modes_many_of_both_launches():
    shapes = [(900, 20), (900, 200), (70, 9), (1200, 150)]
    hs = [S.sdmd_create(n, m, S.SDMD_U8) for n, m in shapes]
    r = [6] * len(hs)
    lam = torch.zeros((2, len(hs), 6), dtype=torch.complex128, device="cuda")
    rank = torch.zeros((2, len(hs)), dtype=torch.int32, device="cuda")
    try:
        for h, (n, m) in zip(hs, shapes):
            S.sdmd_push_batch(h, m, _u8(m, n, n), n)
        S.sdmd_modes_many(hs, r, list(lam[0]), rank[0])
        graph = _replay(lambda st: S.sdmd_modes_many(hs, r, list(lam[1]), rank[1], st))
        assert torch.equal(*torch.view_as_real(lam)) and torch.equal(*rank)
        del graph
    finally:
        for h in hs:
            S.sdmd_destroy(h)
