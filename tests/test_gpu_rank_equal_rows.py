"""Rankings of more scores than are formed at a time (1 GiB): equal stored rows in the
first and in the last part have equal scores and rank by row number, and the scores
are those of one dense call. The sizes are such that the last part alone would divide
its sums over the coordinates differently from the others (152 SMs)."""
import pytest
import torch

from paper_2609_37842_gb300 import eogp as E

pytestmark = pytest.mark.gpu
N, Q = 270000, 1024  # parts of 254,144 rows


def check(train, ts, ks, mode, query):
    v, i = E.score_topk(train, ts, ks, mode, query, 4)
    dense = E.score(train, ts, ks, mode, query)
    E.sync_status()
    q = torch.arange(Q, device="cuda")
    assert torch.equal(i[:, 0].long(), 5 + q)
    assert torch.equal(i[:, 1].long(), N - Q + q)
    assert torch.equal(v[:, 0], v[:, 1])
    assert torch.equal(torch.gather(dense, 1, i.long()), v)


def test_paper():
    g = torch.Generator("cuda").manual_seed(1)
    ks = [1024] * 12
    train = torch.randint(-2 ** 31, 2 ** 31 - 1, (N, 384), device="cuda", generator=g, dtype=torch.int32)
    ts = torch.exp(0.5 * torch.randn((N, 12), device="cuda", generator=g)).clamp(max=3.0)
    train[N - Q:], ts[5:5 + Q] = train[5:5 + Q], 3.0
    ts[N - Q:] = ts[5:5 + Q]
    bits = ((train[5:5 + Q, :, None] >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1).reshape(Q, -1)
    query = (2 * bits - 1).float() * torch.rand((Q, 12288), device="cuda", generator=g)
    check(train, ts, ks, E.SCORE_PAPER, query)


def test_fp():
    g = torch.Generator("cuda").manual_seed(2)
    train = torch.randn((N, 8192), device="cuda", generator=g)
    train[N - Q:] = train[5:5 + Q]
    query = train[5:5 + Q] + 0.1 * torch.randn((Q, 8192), device="cuda", generator=g)
    check(train, None, [8192], E.SCORE_FP, query)
