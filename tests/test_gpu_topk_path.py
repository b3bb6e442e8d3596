"""Ranking 1024 queries over millions of rows of one wide module: the default takes
the fused path from 2,500,000 rows on, the dense one below, with the same lists."""
import pytest
import torch

from paper_2609_37842_gb300 import eogp as E

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,Q,fused", [(2499999, 1024, False), (2500000, 1023, False), (2500001, 1024, True)])
def test_default_path(N, Q, fused):
    g = torch.Generator("cuda").manual_seed(N + Q)
    bits = lambda n: torch.randint(-2 ** 31, 2 ** 31 - 1, (n, 512), generator=g, device="cuda", dtype=torch.int32)
    train, query = bits(N), bits(Q)
    train[N - 1] = query[Q - 1]  # the best row of the last query is the last one
    ts, qs = (0.5 + torch.rand((n, 1), generator=g, device="cuda") for n in (N, Q))
    assert (E.score_topk_workspace_size(N, [16384], E.SCORE_CODES, Q, 20) < 2 ** 29) == fused
    got = E.score_topk(train, ts, [16384], E.SCORE_CODES, query, 20, query_scales=qs)
    with E.options(topk_path=2):
        want = E.score_topk(train, ts, [16384], E.SCORE_CODES, query, 20, query_scales=qs)
    E.sync_status()
    assert all(torch.equal(x, y) for x, y in zip(got, want))
    assert int(got[1][Q - 1, 0]) == N - 1
