"""Unquantised scores that rest on one or two coordinates, where no sum hides a dropped
product of the three-way split, and on values so small that bf16 cannot hold their
third part, at every query tile width.

Bounds. Every product is formed to 2^-30 of itself. One coordinate: nothing else is
added, so one rounding to fp32, 2^-24, and 2^-29 for the roundings of the lower parts'
sum. Two: besides, the tensor core adds two products of the largest parts, with at
least 24 bits, 2^-23. In fp32's subnormal range the rounding unit is 2^-149; there are
eight products a coordinate."""
import numpy as np
import pytest
import torch

from paper_2609_37842_gb300 import eogp as E

pytestmark = pytest.mark.gpu
N, D = 700, 1024


def rows(rng, nz, ex):
    x = np.zeros((N, D))
    for r in range(N):
        x[r, rng.choice(D, nz, replace=False)] = rng.standard_normal(nz) * 2.0 ** ex
    return x.astype(np.float32)


@pytest.mark.parametrize("Q", [3, 17, 33, 64, 130])
@pytest.mark.parametrize("nz,ex,ey", [(1, 0, 0), (2, 0, 0), (1, -100, 0), (1, -104, 0), (1, -112, 3), (1, -118, 30), (2, -125, 60),
                                      (1, -135, 90), (1, 60, -120), (2, 50, -128)])
def test_products(Q, nz, ex, ey):
    rng = np.random.default_rng(abs(1000 * nz + 10 * ey - ex + Q))
    x, y = rows(rng, nz, ex), (rng.standard_normal((Q, D)) * 2.0 ** ey).astype(np.float32)
    got = E.score(torch.from_numpy(x).cuda(), None, [D], E.SCORE_FP, torch.from_numpy(y).cuda())
    E.sync_status()
    got = got.cpu().numpy().astype(np.float64)
    x, y = x.astype(np.float64), y.astype(np.float64)
    bar = (2.0 ** -24 + 2.0 ** -29 + (2.0 ** -23 if nz > 1 else 0.0)) * (np.abs(y) @ np.abs(x).T) + 8 * nz * 2.0 ** -149
    assert np.all(np.abs(got - y @ x.T) <= bar)


def test_tiny_values_beside_others():
    """A row or query with such a value gives the same scores as one fp32 chain."""
    rng = np.random.default_rng(5)
    x, y = (rng.integers(-4, 5, (n, D)).astype(np.float32) for n in (N, 50))
    x[3, 5], x[640, 100], y[49, 9] = 3e-39, -1.0000001e-36, 7e-42
    X, Y = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    got = E.score(X, None, [D], E.SCORE_FP, Y)
    chain = E.score(X, None, [D], E.SCORE_FP, Y, ws=torch.empty(0, dtype=torch.uint8, device="cuda"))
    E.sync_status()
    assert torch.equal(got, chain)
