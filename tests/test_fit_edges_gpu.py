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
