"""Calls whose kernel depends on sizes, alignment or where their buffers lie,
each against the call's other route or a plain reference:

* sdmd_push_batch, sdmd_push_many and sdmd_modes_many with aligned, unaligned
  and host buffers: the same G and eigenvalues bit for bit;
* sdmd_modes (windows from 72 pairs on lie over a cluster of CTAs) against
  sdmd_modes_many (one CTA per window up to 144 pairs), bit for bit;
* Phi and the POD modes at tile edges, odd n and every mode tile;
* Fourier-sparse rows around the chunk length; the uint8 Gram over enough
  positions that the 32-bit sums are flushed.
"""
import numpy as np
import pytest
import torch

from paper_1612_07875_gb300 import sdmd as S

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
KIND = {"u8": (S.SDMD_U8, torch.int64), "f32": (S.SDMD_F32, torch.float64), "c64": (S.SDMD_C64, torch.complex128)}


def _frames(kind, count, n, seed):
    rng = np.random.default_rng(seed)
    if kind == "u8":
        return rng.integers(0, 256, (count, n), dtype=np.uint8)
    x = rng.standard_normal((count, n), dtype=np.float32)
    if kind == "c64":
        x = (x + 1j * rng.standard_normal((count, n), dtype=np.float32)).astype(np.complex64)
    return x


def _gram(h, c, kind):
    G = torch.zeros((c, c), dtype=KIND[kind][1], device="cuda")
    S.sdmd_gram(h, G)
    return torch.view_as_real(G) if G.is_complex() else G


def _offset(x, elems):
    """x on the GPU, starting `elems` elements into its allocation."""
    buf = torch.zeros(x.size + elems, dtype=torch.from_numpy(x[..., :1].copy()).dtype, device="cuda")
    buf[elems:] = torch.from_numpy(x.reshape(-1).copy()).cuda()
    return buf[elems:]


@pytest.mark.parametrize("kind,n,pad,off", [("u8", 1, 0, 0), ("u8", 17, 3, 1), ("u8", 40013, 0, 5), ("u8", 65536, 16, 0),
                                            ("u8", 200003, 13, 15), ("f32", 5, 1, 1), ("f32", 30001, 2, 3)])
def test_push_batch_sources(kind, n, pad, off):
    m, k = 12, 9
    x = _frames(kind, k + m, n + pad, n + off)
    hs = [S.sdmd_create(n, m, KIND[kind][0]) for _ in range(2)]
    try:
        for h in hs:
            S.sdmd_push_batch(h, m, x[:m].copy(), n + pad)
        S.sdmd_push_batch(hs[0], k, _offset(x[m:], off), n + pad)
        S.sdmd_push_batch(hs[1], k, x[m:].copy(), n + pad)
        for _ in range(2):
            assert torch.equal(_gram(hs[0], m, kind), _gram(hs[1], m, kind))
            for h in hs:
                S.sdmd_rebuild(h)      # the same slots
        if kind == "u8":
            w = x[-m:, :n].astype(np.int64)
            assert np.array_equal(_gram(hs[0], m, kind).cpu().numpy(), w @ w.T)
        assert all(S.sdmd_status(h) == S.SDMD_OK for h in hs)
    finally:
        for h in hs:
            S.sdmd_destroy(h)


@pytest.mark.parametrize("off", [0, 1, 4])
def test_push_many_and_modes_many_buffers(off):
    shapes = [("u8", 30011, 9), ("f32", 1, 3), ("u8", 7, 66), ("c64", 513, 5), ("f32", 65541, 20)]
    sets = [[S.sdmd_create(n, m, KIND[k][0]) for k, n, m in shapes] for _ in range(2)]
    try:
        data = [_frames(k, m + 2, n, i + off) for i, (k, n, m) in enumerate(shapes)]
        for t in range(70):
            at = [i for i, (_, _, m) in enumerate(shapes) if t < m + 2]
            if at:
                S.sdmd_push_many([sets[0][i] for i in at], [_offset(data[i][t], off) for i in at])
                S.sdmd_push_many([sets[1][i] for i in at], [data[i][t].copy() for i in at])
                torch.cuda.synchronize()
        for (k, _, m), a, b in zip(shapes, *sets):
            assert torch.equal(_gram(a, m, k), _gram(b, m, k))
        real = [i for i, s in enumerate(shapes) if s[0] != "c64"]
        r = [min(4, shapes[i][2] - 1) for i in real]
        dev = [torch.zeros(q, dtype=torch.complex128, device="cuda") for q in r]
        pin = [torch.zeros(q, dtype=torch.complex128).pin_memory() for q in r]
        rd, rp = torch.zeros(len(r), dtype=torch.int32, device="cuda"), torch.zeros(len(r), dtype=torch.int32).pin_memory()
        S.sdmd_modes_many([sets[0][i] for i in real], r, dev, rd)
        S.sdmd_modes_many([sets[1][i] for i in real], r, pin, rp)
        same = [torch.zeros(max(r), dtype=torch.complex128, device="cuda")] * len(r)   # one buffer: the last handle's stay
        S.sdmd_modes_many([sets[1][i] for i in real], r, same)
        torch.cuda.synchronize()
        assert torch.equal(rd.cpu(), rp)
        for a, b in zip(dev, pin):
            assert torch.equal(torch.view_as_real(a).cpu(), torch.view_as_real(b))
        assert torch.equal(torch.view_as_real(same[0][:r[-1]]).cpu(), torch.view_as_real(pin[-1]))
    finally:
        for h in sets[0] + sets[1]:
            S.sdmd_destroy(h)


@pytest.mark.parametrize("m,r,kind", [(72, 10, "u8"), (73, 10, "u8"), (74, 3, "f32"), (75, 40, "u8"), (80, 79, "f32"),
                                      (100, 10, "u8"), (121, 24, "f32"), (144, 33, "u8"), (145, 10, "f32")])
def test_cluster_window_alone_equals_one_cta(m, r, kind):
    n = 900
    h = S.sdmd_create(n, m, KIND[kind][0])
    try:
        S.sdmd_push_batch(h, m, _frames(kind, m, n, m + r), n)
        lam = torch.zeros((2, r), dtype=torch.complex128, device="cuda")
        sig = torch.zeros((2, r), dtype=torch.float64, device="cuda")
        V = torch.zeros((2, r, m - 1), dtype=torch.float64, device="cuda")
        ranks = torch.zeros(2, dtype=torch.int32, device="cuda")
        S.sdmd_modes(h, r, None, lam[0], ranks[:1])
        S.sdmd_svd(h, r, sig[0], V[0])
        S.sdmd_modes_many([h], [r], [lam[1]], ranks[1:])
        S.sdmd_svd(h, r, sig[1], V[1])
        for a in (torch.view_as_real(lam), sig, V, ranks):
            assert torch.equal(a[0], a[1])
        assert S.sdmd_status(h) == S.SDMD_OK and int(ranks[0]) > 0
    finally:
        S.sdmd_destroy(h)


# n: below one tile, a tile and one more or less for every positions-per-tile,
# the sizes where all modes fit one pass; r: every mode tile and a remainder pass
@pytest.mark.parametrize("kind", ["u8", "f32", "c64"])
@pytest.mark.parametrize("n,r,off", [(67, 1, 0), (511, 3, 1), (513, 5, 0), (1023, 8, 0), (1025, 10, 1), (2047, 11, 0),
                                     (2049, 14, 0), (4097, 16, 0), (40003, 10, 1), (80000, 17, 0), (160001, 4, 0),
                                     (300007, 12, 0)])
def test_phi_and_pod_tiles(kind, n, r, off):
    m = r + 5
    x = _frames(kind, m, n, n + r)
    h = S.sdmd_create(n, m, KIND[kind][0])
    try:
        S.sdmd_push_batch(h, m, x.copy(), n)
        S.sdmd_set_option(h, S.SDMD_OPT_PHI_TENSOR, 0)
        buf = torch.full((r * n + off,), float("nan"), dtype=torch.complex64, device="cuda")
        lam = torch.zeros(r, dtype=torch.complex128, device="cuda")
        S.sdmd_modes(h, r, buf[off:], lam)
        phi = buf[off:].cpu().numpy().reshape(r, n).T.astype(np.complex128)
        # Phi = X' M: each entry is p products and sums in FP32 of the same M, so
        # the least-squares residual of a column is below that of the true M
        # (M rounded once: 2^-24 of |x||m|; complex data: four products an entry)
        X = x[1:].T.astype(np.complex128 if kind == "c64" else np.float64)
        p = m - 1
        M = np.linalg.lstsq(X, phi, rcond=None)[0]
        bound = (4 * p + 4) * U * np.linalg.norm(np.abs(X) @ np.abs(M), axis=0)
        assert np.isfinite(phi).all()
        assert (np.linalg.norm(phi - X @ M, axis=0) <= 1.01 * bound).all()
        if kind != "c64":
            sig = torch.zeros(r, dtype=torch.float64, device="cuda")
            V = torch.zeros((r, p), dtype=torch.float64, device="cuda")
            S.sdmd_svd(h, r, sig, V)
            Ub = torch.full((r * n + off,), float("nan"), dtype=torch.float32, device="cuda")
            S.sdmd_pod_modes(h, r, Ub[off:])
            W = (V / sig[:, None]).cpu().numpy().T
            X0 = x[:-1].T.astype(np.float64)
            err = np.abs(Ub[off:].cpu().numpy().reshape(r, n).T - X0 @ W)
            assert (err <= (p + 2) * 1.01 * U * (np.abs(X0) @ np.abs(W))).all()
        assert S.sdmd_status(h) == S.SDMD_OK
    finally:
        S.sdmd_destroy(h)


@pytest.mark.parametrize("device", [True, False])
@pytest.mark.parametrize("nnz", [[1, 2, 0, 9], [2047, 2048, 2049, 7], [255, 256, 257, 4097], [6000, 5999, 1, 2056]])
def test_sparse_row_chunks(device, nnz):
    n, m = 20000, 4
    rng = np.random.default_rng(sum(nnz))
    h = S.sdmd_create_sparse(n, m, 6000)
    dense = np.zeros((2 * m, n), dtype=np.complex128)
    try:
        for t in range(2 * m):
            k = nnz[t % m]
            idx = np.sort(rng.choice(n, k, replace=False)).astype(np.int32)
            val = (rng.standard_normal(k) + 1j * rng.standard_normal(k)).astype(np.complex64)
            dense[t, idx] = val
            if device:
                S.sdmd_push_sparse(h, k, torch.from_numpy(idx).cuda(), torch.from_numpy(val).cuda())
            else:
                S.sdmd_push_sparse(h, k, idx, val)
        G = torch.zeros((m, m), dtype=torch.complex128, device="cuda")
        S.sdmd_gram(h, G)
        D = dense[m:]
        ref, scale = D.conj() @ D.T, np.abs(D) @ np.abs(D).T
        # FP32 products (two an entry and part), a thread's sum of at most 8
        # entries (16 additions) before FP64
        assert (np.abs(G.cpu().numpy() - ref) <= 2 * 20 * U * scale + 1e-300).all()
        assert S.sdmd_status(h) == S.SDMD_OK
    finally:
        S.sdmd_destroy(h)


@pytest.mark.parametrize("n,lo", [(127, 0), (2049, 0), (4096 * 152 + 255, 1), ((1 << 23) + 5, 0)])
def test_u8_gram_flush(n, lo):
    m = 4
    h = S.sdmd_create(n, m, S.SDMD_U8)
    try:
        x = torch.full((m, n), 255, dtype=torch.uint8, device="cuda")
        x[1] = lo
        x[2, n // 2:] = 0
        x[3, ::2] = 3
        torch.cuda.synchronize()
        S.sdmd_push_batch(h, m, x, n)
        w = x.cpu().numpy().astype(np.int64)
        ref = w @ w.T
        assert np.array_equal(_gram(h, m, "u8").cpu().numpy(), ref)
        S.sdmd_rebuild(h)
        assert np.array_equal(_gram(h, m, "u8").cpu().numpy(), ref)
    finally:
        S.sdmd_destroy(h)
