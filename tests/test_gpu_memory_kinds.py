"""Buffers that are not this GPU's own memory. A kernel may touch another
GPU's memory only with peer access, so snapshots, Gram matrices and rows that
lie elsewhere are moved by copies. Managed memory takes the same route as
another GPU's and exists on one GPU: the calls are captured into a graph and
have to hold copy nodes for it (none for this GPU's memory), and the results
are those of plain device buffers."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1612_07875_gb300 import sdmd as S

pytestmark = pytest.mark.gpu

KERNEL, MEMCPY = 0, 1                  # CUgraphNodeType


def _driver():
    return ctypes.CDLL("libcuda.so.1")


def _ok(rc):
    assert rc == 0, "CUresult %d" % rc


class Managed:
    """A managed allocation holding a copy of `a`."""

    def __init__(self, a):
        self.d, self.a = _driver(), np.ascontiguousarray(a)
        p = ctypes.c_uint64()
        _ok(self.d.cuMemAllocManaged(ctypes.byref(p), ctypes.c_size_t(self.a.nbytes), ctypes.c_uint(1)))
        self.ptr = p.value
        ctypes.memmove(self.ptr, self.a.ctypes.data, self.a.nbytes)

    def read(self):
        torch.cuda.synchronize()
        out = np.empty_like(self.a)
        ctypes.memmove(out.ctypes.data, self.ptr, out.nbytes)
        return out

    def free(self):
        torch.cuda.synchronize()
        _ok(self.d.cuMemFree_v2(ctypes.c_uint64(self.ptr)))


def _nodes(call):
    """Types of the graph nodes that `call(stream)` enqueues (nothing runs)."""
    d, st = _driver(), torch.cuda.Stream()
    torch.cuda.synchronize()
    raw, g = ctypes.c_void_p(st.cuda_stream), ctypes.c_void_p()
    _ok(d.cuStreamBeginCapture_v2(raw, ctypes.c_int(2)))
    try:
        call(st)
    finally:
        rc = d.cuStreamEndCapture(raw, ctypes.byref(g))
    _ok(rc)
    n = ctypes.c_size_t()
    _ok(d.cuGraphGetNodes(g, None, ctypes.byref(n)))
    nodes, types = (ctypes.c_void_p * n.value)(), []
    _ok(d.cuGraphGetNodes(g, nodes, ctypes.byref(n)))
    for node in nodes:
        t = ctypes.c_int()
        _ok(d.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(t)))
        types.append(t.value)
    _ok(d.cuGraphDestroy(g))
    return types


@pytest.mark.parametrize("n", [4096, 1003])
def test_managed_buffers_go_through_copies(n):
    m = 5
    rng = np.random.default_rng(n)
    x = rng.standard_normal((m, n), dtype=np.float32)
    dev = torch.from_numpy(x).cuda()
    man = [Managed(r) for r in x]
    batch, Gm = Managed(x[:2].copy()), Managed(np.zeros((m, m)))
    row = Managed(np.zeros(m))
    hs = [S.sdmd_create(n, m, S.SDMD_F32) for _ in range(3)]
    piped = S.sdmd_create_ex(n, m, S.SDMD_F32, 2)
    G = torch.zeros((m, m), dtype=torch.float64, device="cuda")
    try:
        S.sdmd_push_batch(hs[0], m, dev, n)
        S.sdmd_push_batch(hs[1], 2, batch.ptr, n)
        S.sdmd_push(hs[1], man[2].ptr)
        S.sdmd_push_many([hs[1]], [man[3].ptr])
        S.sdmd_push(hs[1], man[4].ptr)
        S.sdmd_gram(hs[0], G)
        S.sdmd_gram(hs[1], Gm.ptr)
        ref = G.cpu().numpy()
        assert np.array_equal(Gm.read(), ref)
        S.sdmd_newest_row(hs[1], row.ptr)
        assert np.array_equal(row.read(), ref[-1])
        S.sdmd_set_newest_row(hs[1], row.ptr)
        S.sdmd_gram(hs[1], Gm.ptr)
        assert np.array_equal(Gm.read(), ref)
        h = hs[2]
        S.sdmd_push(h, dev[0])
        cases = [("push", lambda p, st: S.sdmd_push(h, p, st), man[0].ptr, dev[0]),
                 ("push_batch", lambda p, st: S.sdmd_push_batch(h, 2, p, n, st), batch.ptr, dev),
                 ("push_many", lambda p, st: S.sdmd_push_many([h], [p], st), man[0].ptr, dev[0]),
                 ("step", lambda p, st: S.sdmd_step(piped, p, 2, None, None, None, st), man[0].ptr, dev[0]),
                 ("gram", lambda p, st: S.sdmd_gram(h, p, st), Gm.ptr, G),
                 ("newest_row", lambda p, st: S.sdmd_newest_row(h, p, st), row.ptr, G[0]),
                 ("set_newest_row", lambda p, st: S.sdmd_set_newest_row(h, p, st), row.ptr, G[0])]
        for name, call, managed, device in cases:
            assert MEMCPY in _nodes(lambda st: call(managed, st)), name
            if n % 4 == 0:                               # (rows off 16 bytes are copied wherever they lie)
                assert MEMCPY not in _nodes(lambda st: call(device, st)), name
    finally:
        for q in hs + [piped]:
            S.sdmd_destroy(q)
        for b in man + [batch, Gm, row]:
            b.free()
