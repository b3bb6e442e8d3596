"""Unquantised scores beside a row or a query with a NaN, an infinity or a value too
small for the tensor cores' split keep their bits: equal rows have equal scores and
rank by row number wherever such a value stands."""
import pytest
import torch

from paper_2609_37842_gb300 import eogp as E

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), 1.0000001e-38])
@pytest.mark.parametrize("N,Q,D", [(300, 70, 2048), (1000, 5, 12288), (129, 20, 520)])
def test_neighbours_keep_their_bits(N, Q, D, bad):
    g = torch.Generator("cuda").manual_seed(N)
    x, y = (torch.randn((n, D), device="cuda", generator=g) for n in (N, Q))
    clean = E.score(x, None, [D], E.SCORE_FP, y)
    rows, queries = [0, 70, N - 1], [Q - 2]
    x[rows, 17] = bad
    y[queries, D - 1] = bad
    got = E.score(x, None, [D], E.SCORE_FP, y)
    chain = E.score(x, None, [D], E.SCORE_FP, y, ws=torch.empty(0, dtype=torch.uint8, device="cuda"))
    E.sync_status()
    noted = torch.zeros((Q, N), dtype=torch.bool, device="cuda")
    noted[:, rows] = True
    noted[queries] = True
    assert torch.equal(got[~noted], clean[~noted])
    assert torch.equal(got[noted].nan_to_num(nan=7.5), chain[noted].nan_to_num(nan=7.5))


def test_equal_rows_rank_by_number():
    g = torch.Generator("cuda").manual_seed(9)
    N, Q, D = 1000, 40, 4096
    x = torch.randn((N, D), device="cuda", generator=g)
    x[900:940] = x[100:140]
    y = x[100:140] + 0.1 * torch.randn((Q, D), device="cuda", generator=g)
    x[127, 3], x[950, 0] = float("nan"), float("nan")  # in a tile with the first, and with the second copies
    x[927] = x[127]
    v, i = E.score_topk(x, None, [D], E.SCORE_FP, y, 2)
    E.sync_status()
    q = torch.tensor([r for r in range(Q) if r != 27], device="cuda")
    assert torch.equal(i[q, 0].long(), 100 + q) and torch.equal(i[q, 1].long(), 900 + q)
    assert torch.equal(v[q, 0], v[q, 1])
