"""Windows whose G_X lies over a cluster (more than 144 snapshot pairs), alone
and batched with short windows, against the FP64 eigenvalues of the handle's
own G; and the same handle's batched results equal to its own bit for bit.
Sizes: the last one-CTA window, the first cluster windows, lengths with every
remainder of the row classes, the longest window, r up to more Ritz vectors
than fit on chip."""
import numpy as np
import pytest
import torch

from paper_1612_07875_gb300 import sdmd as S

pytestmark = pytest.mark.gpu


def _handle(n, m, seed):
    rng = np.random.default_rng(seed)
    x = rng.integers(0, 256, (m, n), dtype=np.uint8)
    h = S.sdmd_create(n, m, S.SDMD_U8)
    for row in x:
        S.sdmd_push(h, torch.from_numpy(row).cuda())
    x = x.astype(np.int64)
    return h, (x @ x.T).astype(np.float64)


@pytest.mark.parametrize("m,r", [(145, 10), (146, 10), (147, 5), (150, 30), (153, 60), (200, 10), (256, 10), (256, 255)])
def test_cluster_windows(m, r):
    h, g = _handle(3000, m, m + r)
    hs, _ = _handle(2000, 24, 5)
    try:
        lam = torch.zeros(r, dtype=torch.complex128, device="cuda")
        sigma = torch.zeros(r, dtype=torch.float64, device="cuda")
        V = torch.zeros((r, m - 1), dtype=torch.float64, device="cuda")
        S.sdmd_modes(h, r, None, lam)
        S.sdmd_svd(h, r, sigma, V)
        assert S.sdmd_status(h) == S.SDMD_OK
        ref = np.linalg.eigvalsh(g[:m - 1, :m - 1])[::-1][:r]
        # df64 backward error of the eigensolver: about 1e-13 lambda_1
        assert np.abs(sigma.cpu().numpy() ** 2 - ref).max() <= 1e-12 * ref[0]
        v = V.cpu().numpy()
        assert np.abs(v @ v.T - np.eye(r)).max() <= 1e-10
        out = [torch.zeros(r, dtype=torch.complex128, device="cuda"), torch.zeros(5, dtype=torch.complex128, device="cuda")]
        S.sdmd_modes_many([h, hs], [r, 5], out)
        alone = torch.zeros(5, dtype=torch.complex128, device="cuda")
        S.sdmd_modes(hs, 5, None, alone)
        assert torch.equal(torch.view_as_real(out[0]), torch.view_as_real(lam))
        assert torch.equal(torch.view_as_real(out[1]), torch.view_as_real(alone))
    finally:
        S.sdmd_destroy(h)
        S.sdmd_destroy(hs)
