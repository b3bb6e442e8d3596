"""Unquantised scores and rankings of the most queries a call may have: the last sizes
whose whole query tiles are 65,472 and 65,536 queries. Integer coordinates, so every
kernel gives the same sums."""
import pytest
import torch

from paper_2609_37842_gb300 import eogp as E

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Q", [65472, 65473, 65500, 65535])
def test_fp_many_queries(Q):
    g = torch.Generator("cuda").manual_seed(Q)
    N, D = 131, 512
    x, y = (torch.randint(-4, 5, (n, D), device="cuda", generator=g).float() for n in (N, Q))
    want = y @ x.t()  # integers below 2^24
    got = E.score(x, None, [D], E.SCORE_FP, y)
    v, i = E.score_topk(x, None, [D], E.SCORE_FP, y, 3)
    E.sync_status()
    assert torch.equal(got, want)
    assert torch.equal(v, want.topk(3, dim=1).values)
    assert torch.equal(torch.gather(want, 1, i.long()), v)
