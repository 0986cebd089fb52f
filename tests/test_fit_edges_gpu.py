"""The one-launch eigen-solver of the fits at the sizes where its split can go wrong: two indices, block counts that leave columns
over, the largest cluster, the register tiles' limits, the two-sided solver beyond it, rank-deficient and all-zero data.

The eigen-pairs are checked against the matrix itself, in fp64: || C u - lambda u || and the spectrum within 1e-11 of the largest
eigenvalue (n eps with a margin of 100; the solver stops at cosines of 1e-10 before its last rotations), orthonormality within
2e-6 (the output's rounding to fp32, 6e-8 per entry, over sqrt(n) entries).
"""
import numpy as np
import pytest
import torch

from paper_2605_16439_b200 import binding as kvc
from paper_2605_16439_b200 import build as kvc_build
from paper_2605_16439_b200 import workloads as wl

import kvc_testlib as tl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    kvc_build.build()


@pytest.mark.parametrize("n,B,H", [(2, 1, 1), (3, 1, 2), (17, 2, 3), (33, 1, 2), (65, 1, 1), (129, 2, 2), (255, 2, 2), (257, 3, 1), (400, 4, 1),
                                   (640, 5, 1), (642, 6, 1), (100, 0, 2)])
def test_eigenpairs(n, B, H):
    gen = torch.Generator().manual_seed(n)
    V = torch.randn((max(B, 1), H, n, 128), generator=gen)
    if B == 0:
        V = V[..., :1].expand(-1, -1, -1, 128).contiguous()          # one column repeated: rank one
    U, mu, eig, sweeps = kvc.kvc_fit_value_pca(V.to(DEV), n, n, want_eig=True)
    assert 0 < sweeps < 40
    U, eig, V64 = tl.np64(U), eig.cpu().numpy(), tl.np64(V)
    for h in range(H):
        X = V64[:, h] - V64[:, h].reshape(-1, 128).mean(axis=0)
        C = np.einsum("bnc,bmc->nm", X, X)
        want = np.linalg.eigvalsh(C)[::-1]
        np.testing.assert_allclose(eig[h], want, atol=1e-11 * want[0])
        np.testing.assert_allclose(U[h] @ U[h].T, np.eye(n), atol=2e-6)
        np.testing.assert_allclose(U[h] @ C, eig[h][:, None] * U[h], atol=2e-6 * want[0])


def test_all_zero_samples():
    U, mu, eig, sweeps = kvc.kvc_fit_value_pca(torch.zeros((1, 2, 20, 128), device=DEV), 20, 7, want_eig=True)
    assert (eig == 0).all() and (mu == 0).all() and sweeps < 40
    np.testing.assert_allclose(tl.np64(U)[0] @ tl.np64(U)[0].T, np.eye(7), atol=2e-6)


def test_samples_at_an_unaligned_address():
    raw = torch.randn(2 * 36 * 128 + 1, device=DEV)
    V = raw[1:].view(1, 2, 36, 128)
    a = kvc.kvc_fit_value_pca(V, 36, 10, want_eig=True)
    b = kvc.kvc_fit_value_pca(V.clone(), 36, 10, want_eig=True)
    assert torch.equal(a[0], b[0]) and torch.equal(a[2], b[2])


def _clustered(kind, gen):
    """[B, 1, n, 128] samples whose token covariance has many eigenvalues close to one another."""
    if kind == "one block":            # fewer samples than positions: a null space of 68, 128 or 272
        return wl.vision_kv(1, 1, 1, 14, 128, 7).view(1, 1, 196, 128)
    if kind == "one block of 256":
        return wl.vision_kv(1, 1, 1, 16, 128, 7).view(1, 1, 256, 128)
    if kind == "one block of 400":
        return wl.vision_kv(1, 1, 1, 20, 128, 7).view(1, 1, 400, 128)
    if kind == "repeated rows":        # every position four times, up to 1e-6
        return (torch.randn((1, 1, 64, 128), generator=gen).repeat_interleave(4, dim=2) +
                1e-6 * torch.randn((1, 1, 256, 128), generator=gen))
    if kind == "parallel rows":        # eight directions, lengths between 0.1 and 10
        return torch.randn((1, 1, 8, 128), generator=gen).repeat_interleave(25, dim=2) * (0.1 + 9.9 * torch.rand((1, 1, 200, 1), generator=gen))
    # eigenvalues equal to 1e-5: columns orthonormal and orthogonal to the ones, so that the mean is zero
    n = 128
    X = torch.randn((n, n - 1), generator=gen, dtype=torch.float64)
    Q = torch.linalg.qr(X - X.mean(dim=0))[0] * (1 + 5e-6 * torch.rand((1, n - 1), generator=gen, dtype=torch.float64))
    return torch.nn.functional.pad(Q, (0, 129 - n)).float().view(1, 1, n, 128)


@pytest.mark.parametrize("kind", ["one block", "one block of 256", "one block of 400", "repeated rows", "parallel rows", "close"])
def test_clustered_eigenvalues(kind):
    """Where eigenvalues cluster the cosines fall by a factor of ten a sweep, not quadratically: the solver goes on until they are gone.

    Orthonormality: entries of two unit rows rounded to fp32, 2^-24 of each, change their product by at most 2^-23; spectrum as above."""
    V = _clustered(kind, torch.Generator().manual_seed(11))
    n = V.shape[2]
    U, mu, eig, sweeps = kvc.kvc_fit_value_pca(V.to(DEV), n, n, want_eig=True)
    assert 0 < sweeps < 40
    U, X = tl.np64(U)[0], tl.np64(V)[0, 0]
    X = X - X.mean(axis=0)
    want = np.linalg.eigvalsh(X @ X.T)[::-1]
    np.testing.assert_allclose(eig.cpu().numpy()[0], want, atol=1e-11 * want[0])
    np.testing.assert_allclose(U @ U.T, np.eye(n), atol=1.01 * 2.0 ** -23)
