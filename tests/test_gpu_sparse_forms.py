"""The Fourier-sparse row takes a thread's entries one after the other, together,
or with the values loaded ahead of the tags, by the size of the lookup tables
and of the launch. The sums are the same in the same order: handles that differ
only in n, so in the form, hold the same G bit for bit."""
import numpy as np
import pytest
import torch

from paper_1612_07875_gb300 import sdmd as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nnz,m,shared", [(1, 3, 1.0), (2049, 5, 0.5), (6000, 4, 0.0), (15_000, 90, 0.9)])
def test_forms_agree(nnz, m, shared):
    rng = np.random.default_rng(nnz)
    top = 100_000
    sizes = [top, (1 << 22) + 1, (1 << 25) + 1]           # ahead or together; together; one after the other
    hs = [S.sdmd_create_sparse(n, m, nnz) for n in sizes]
    common = rng.choice(top, nnz, replace=False)
    dense = np.zeros((m, top), dtype=np.complex128)
    try:
        for t in range(m + 1):
            keep = int(shared * nnz)
            idx = np.unique(np.concatenate([common[:keep], rng.choice(top, nnz - keep, replace=False)]))[:nnz].astype(np.int32)
            val = (rng.standard_normal(idx.size) + 1j * rng.standard_normal(idx.size)).astype(np.complex64)
            dense[t % m] = 0
            dense[t % m, idx] = val
            di, dv = torch.from_numpy(idx).cuda(), torch.from_numpy(val).cuda()
            for h in hs:
                S.sdmd_push_sparse(h, idx.size, di, dv)
            torch.cuda.synchronize()
        G = [torch.zeros((m, m), dtype=torch.complex128, device="cuda") for _ in hs]
        for h, g in zip(hs, G):
            S.sdmd_gram(h, g)
            assert S.sdmd_status(h) == S.SDMD_OK
        for g in G[1:]:
            assert torch.equal(torch.view_as_real(g), torch.view_as_real(G[0]))
        D = dense[[(t + 1) % m for t in range(m)]]        # oldest first
        ref, scale = D.conj() @ D.T, np.abs(D) @ np.abs(D).T
        # FP32 products (two an entry and part), a thread's sum of at most 8
        # entries (16 additions) before FP64
        assert (np.abs(G[0].cpu().numpy() - ref) <= 2 * 20 * 2.0 ** -24 * scale + 1e-300).all()
    finally:
        for h in hs:
            S.sdmd_destroy(h)
