"""Rankings of so many queries that 1 GiB does not hold their scores of one slice of
rows: the queries go in parts, with the lists that the same queries get in a call of
their own, and the scores' workspace stays at 1 GiB."""
import pytest
import torch

from paper_2609_37842_gb300 import eogp as E

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [E.SCORE_CODES, E.SCORE_PAPER, E.SCORE_FP])
@pytest.mark.parametrize("N,Q", [(33000, 30001), (270, 65535), (17000, 65535)])
def test_query_parts(N, Q, mode):
    g = torch.Generator("cuda").manual_seed(N + mode)
    D = 512 if mode == E.SCORE_FP else 256
    bits = lambda n: torch.randint(-2 ** 31, 2 ** 31 - 1, (n, D // 32), device="cuda", generator=g, dtype=torch.int32)
    ints = lambda n: torch.randint(-3, 4, (n, D), device="cuda", generator=g).float()
    scales = lambda n: torch.randint(1, 5, (n, 1), device="cuda", generator=g).float()
    train = ints(N) if mode == E.SCORE_FP else bits(N)
    ts = None if mode == E.SCORE_FP else scales(N)
    query = bits(Q) if mode == E.SCORE_CODES else ints(Q)
    qs = scales(Q) if mode == E.SCORE_CODES else None
    s, i = E.score_topk(train, ts, [D], mode, query, 5, query_scales=qs)
    for a, b in [(0, 70), (15000, 15060), (16350, 16420), (Q - 70, Q)]:
        s1, i1 = E.score_topk(train, ts, [D], mode, query[a:b], 5, query_scales=None if qs is None else qs[a:b])
        assert torch.equal(s[a:b], s1) and torch.equal(i[a:b], i1)
    E.sync_status()


@pytest.mark.parametrize("N,Q", [(2_000_000, 16384), (2_000_000, 16385), (2_000_000, 20000), (2_000_000, 65535), (16385, 65535), (3, 65535)])
def test_workspace(N, Q):
    K = 20
    lists = 2 * 16448 * 4 * (-(-N // 4096) * K + 8) * 2 if N > 16384 else 0
    assert E.score_topk_workspace_size(N, [1024], E.SCORE_CODES, Q, K) <= 2 ** 30 + lists + 128 * Q * 8 + 4096
