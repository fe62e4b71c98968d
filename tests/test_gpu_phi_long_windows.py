"""Phi and the POD modes of long windows, where a stage holds fewer slots
because M is long, and of short snapshots, in narrow and wide tiles at their
edges and on both sides of the lines between them."""
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


@pytest.mark.parametrize("kind,n,m,r", [("f32", 255, 200, 16), ("f32", 257, 256, 10), ("f32", 1025, 256, 40), ("f32", 58369, 256, 16),
                                        ("f32", 116737, 256, 10), ("f32", 116736, 180, 4), ("f32", 60001, 256, 24),
                                        ("u8", 511, 256, 16), ("u8", 513, 250, 10), ("u8", 40961, 256, 40),
                                        ("c64", 255, 140, 16), ("c64", 257, 100, 10), ("c64", 20001, 140, 24)])
def test_phi_and_pod_of_long_windows(kind, n, m, r):
    x = _frames(kind, m, n, n + r)
    p = m - 1
    h = S.sdmd_create(n, m, KIND[kind][0])
    try:
        S.sdmd_push_batch(h, m, x.copy(), n)
        S.sdmd_set_option(h, S.SDMD_OPT_PHI_TENSOR, 0)
        buf = torch.full((r * n,), float("nan"), dtype=torch.complex64, device="cuda")
        lam = torch.zeros(r, dtype=torch.complex128, device="cuda")
        S.sdmd_modes(h, r, buf, lam)
        phi = buf.cpu().numpy().reshape(r, n).T.astype(np.complex128)
        X = x[1:].T.astype(np.complex128 if kind == "c64" else np.float64)
        # every entry is p products and sums in FP32 of the same M (FP32): the
        # residual of the least-squares M is below that of the true one
        M = np.linalg.lstsq(X, phi, rcond=None)[0]
        bound = (4 * p + 4) * U * np.linalg.norm(np.abs(X) @ np.abs(M), axis=0)
        assert np.isfinite(phi).all()
        if n > p:                              # (fewer positions than slots: any Phi has an exact M)
            assert (np.linalg.norm(phi - X @ M, axis=0) <= 1.01 * bound).all()
        if kind != "c64":
            sig = torch.zeros(r, dtype=torch.float64, device="cuda")
            V = torch.zeros((r, p), dtype=torch.float64, device="cuda")
            S.sdmd_svd(h, r, sig, V)
            Ub = torch.full((r * n,), float("nan"), dtype=torch.float32, device="cuda")
            S.sdmd_pod_modes(h, r, Ub)
            W = (V / sig[:, None]).cpu().numpy().T
            X0 = x[:-1].T.astype(np.float64)
            err = np.abs(Ub.cpu().numpy().reshape(r, n).T - X0 @ W)
            assert (err <= (p + 2) * 1.01 * U * (np.abs(X0) @ np.abs(W))).all()
        assert S.sdmd_status(h) == S.SDMD_OK
    finally:
        S.sdmd_destroy(h)
