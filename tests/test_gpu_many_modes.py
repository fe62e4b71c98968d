"""Eigenvalues of many modes, where H and Q of the Schur iteration are on chip
and the rest of the eigenproblem is not, H alone is, or neither."""
import numpy as np
import pytest
import torch

import oracle
from helpers import match_eigs
from paper_1612_07875_gb300 import sdmd as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,r", [(64, 63), (73, 50), (100, 80), (128, 116), (150, 60), (200, 100), (200, 120), (180, 165)])
def test_many_modes(m, r):
    """FP32 Schur vectors refined by a df64 Rayleigh quotient: an eigenvalue's
    error is second order in the vectors' (2^-24 r), times its condition."""
    n = 3000
    x = np.random.default_rng(m + r).standard_normal((m, n), dtype=np.float32)
    h = S.sdmd_create(n, m, S.SDMD_F32)
    try:
        for row in x:
            S.sdmd_push(h, torch.from_numpy(row).cuda())
        lam = torch.zeros(r, dtype=torch.complex128, device="cuda")
        rank = torch.zeros(1, dtype=torch.int32, device="cuda")
        S.sdmd_modes(h, r, None, lam, rank)
        G = torch.zeros((m, m), dtype=torch.float64, device="cuda")
        S.sdmd_gram(h, G)
        g = G.cpu().numpy()
        ref = oracle.dmd_from_gram(g[:-1, :-1], g[:-1, 1:], r)
        assert int(rank[0]) == ref.r == r
        err, _ = match_eigs(lam.cpu().numpy(), ref.lam)
        assert err <= 1e-6
        assert S.sdmd_status(h) == S.SDMD_OK
    finally:
        S.sdmd_destroy(h)
