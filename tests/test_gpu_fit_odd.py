"""Dense fits whose matrix has an odd number of rows: the index that has no partner in
a Jacobi step still takes the other pairs' rotations. Eigenvalues, and every direction
by itself (its residual in the second moment), in a basis that mixes all columns.
Bounds: the solver stops at an off-diagonal mass of 1e-11 of the matrix's norm, or at
its rounding floor, and directions are written in fp32 (2^-24 an entry)."""
import numpy as np
import pytest
import torch

from paper_2609_37842_gb300 import eogp as E

pytestmark = pytest.mark.gpu


def mixed_rows(n, m):
    rng = np.random.default_rng(n * 7 + m)
    Q, _ = np.linalg.qr(rng.standard_normal((m, m)))
    return ((rng.standard_normal((n, m)) * np.arange(1, m + 1) ** -0.7) @ Q).astype(np.float32)


def check(Pt, eig, C, k):
    Pt, eig = Pt.cpu().numpy().astype(np.float64), eig.cpu().numpy()
    want = np.linalg.eigvalsh(C)[::-1][:k]
    assert np.all(np.abs(eig - want) <= 1e-6 * want[0])
    assert np.abs(Pt @ Pt.T - np.eye(k)).max() <= 1e-5
    # one rounding to fp32 of each entry moves C p by at most 2^-24 ||C||
    assert np.all(np.linalg.norm(Pt @ C - want[:, None] * Pt, axis=1) <= 1e-6 * want[0])


@pytest.mark.parametrize("n,m,k", [(9, 3, 2), (3, 3, 3), (40, 33, 12), (33, 40, 12), (235, 301, 40), (700, 333, 333),
                                   (1100, 1023, 64), (1023, 1200, 64)])
def test_fit_odd(n, m, k):
    Z = mixed_rows(n, m)
    Pt, eig = E.fit_pca(torch.from_numpy(Z).cuda(), k)
    E.sync_status()
    Z = Z.astype(np.float64)
    check(Pt, eig, Z.T @ Z / n, k)


@pytest.mark.parametrize("m,k", [(33, 33), (257, 20)])
def test_fit_odd_from_moment(m, k):
    Z = mixed_rows(500, m).astype(np.float64)
    Pt, eig = E.fit_pca_from_moment(torch.from_numpy(Z.T @ Z).cuda(), 500, k)
    E.sync_status()
    check(Pt, eig, Z.T @ Z / 500, k)
