"""The fit's kernels at the edges of their tiles: sweeps of two pairs and of more
pairs than a warp or a block takes, Cholesky panels and inverse columns of one and of
several blocks (subspace route). Bounds: eigenvalues 1e-6 (dense, fp64 from fp32
inputs) and 1e-3 (subspace, its stopping residual), directions orthonormal to 1e-4."""
import numpy as np
import pytest
import torch

from paper_2609_37842_gb300 import eogp as E

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("n,m,k", [(9, 2, 1), (4, 11, 2), (200, 34, 34), (66, 300, 20), (500, 130, 7), (400, 322, 64),
                                   (1300, 1030, 5), (1100, 1500, 150), (2500, 1200, 257)])
def test_fit_sizes(n, m, k):
    rng = np.random.default_rng(n + m)
    Z = (rng.standard_normal((n, m)) * np.arange(1, m + 1) ** -0.7).astype(np.float32)
    Pt, eig = E.fit_pca(torch.from_numpy(Z).to(DEV), k)
    E.sync_status()
    Pt, eig = Pt.cpu().numpy().astype(np.float64), eig.cpu().numpy()
    Z64 = Z.astype(np.float64)
    C = Z64.T @ Z64 / n
    want = np.linalg.eigvalsh(C)[::-1][:k]
    tol = 1e-6 if min(n, m) <= 1024 else 1e-3
    assert np.all(np.abs(eig - want) <= tol * want[0])
    assert np.abs(Pt @ Pt.T - np.eye(k)).max() <= 1e-4
    # captured energy: the directions hold what their eigenvalues say
    assert abs(np.trace(Pt @ C @ Pt.T) - want.sum()) <= max(tol, 1e-5) * want.sum()
