"""Fits of rows that hold an infinity or a NaN return an error, on every route (dense
of both parities and of one value, Gram, subspace, from a summed moment), write no
directions, and leave the next fit right. (The ranking of the eigenvalues and the
sign rule index by what they find, so they have to hold for any values.)"""
import numpy as np
import pytest
import torch

from paper_2609_37842_gb300 import eogp as E

pytestmark = pytest.mark.gpu
EDEVICE = -6


def rows(n, m):
    g = torch.Generator("cuda").manual_seed(n + m)
    return torch.randn((n, m), device="cuda", generator=g) * torch.arange(1, m + 1, device="cuda") ** -0.7


def clear_status():
    try:
        E.sync_status()
    except E.EOGPError:
        pass


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("n,m,k", [(1, 1, 1), (1, 300, 1), (5, 1, 1), (200, 34, 9), (200, 35, 9), (33, 300, 8),
                                   (1100, 1200, 70), (2000, 1100, 70)])
def test_fit_not_finite(n, m, k, value):
    Z = rows(n, m)
    Z[n // 2, m // 3] = value
    with pytest.raises(E.EOGPError) as e:
        E.fit_pca(Z, k)
    assert e.value.code == EDEVICE
    torch.cuda.synchronize()
    clear_status()
    Z = rows(n, m)
    _, eig = E.fit_pca(Z, k)
    E.sync_status()
    want = torch.linalg.eigvalsh((Z.double().t() @ Z.double() / n).cpu()).flip(0)[:k]
    assert float((eig.cpu().double() - want).abs().max()) <= 1e-3 * float(want[0])


@pytest.mark.parametrize("m,k", [(34, 9), (1100, 70)])
def test_fit_from_moment_not_finite(m, k):
    Z = rows(1500, m)
    C = Z.double().t() @ Z.double()
    C[3, 5] = C[5, 3] = float("nan")
    with pytest.raises(E.EOGPError) as e:
        E.fit_pca_from_moment(C, 1500, k)
    assert e.value.code == EDEVICE
    torch.cuda.synchronize()
    clear_status()
