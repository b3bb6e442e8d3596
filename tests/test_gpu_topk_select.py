"""k_topk_select against the oracle's ranking: rows of one slice and of several,
lengths around the slice and vector edges, and score orders that overflow the
candidate buffer (sorted rows, equal scores), NaN, infinities and signed zeros.
Scores are planted through the FP mode: one query coordinate of 1, stored values as given."""
import numpy as np
import pytest
import torch

from oracle import eogp_oracle as O
from paper_2609_37842_gb300 import eogp as E

pytestmark = pytest.mark.gpu
DEV = "cuda"


def rows(kind, Q, N, rng):
    if kind == "random":
        return rng.standard_normal((Q, N))
    if kind == "descending":      # one thread after another holds all of the best
        return -np.sort(rng.standard_normal((Q, N)), axis=1)
    if kind == "blocks":          # the best scores all in a few threads' places
        x = rng.standard_normal((Q, N))
        x[:, (np.arange(N) // 4) % 512 < 3] += 100.0
        return x
    if kind == "equal":
        return np.zeros((Q, N))
    if kind == "few":             # NaN almost everywhere
        x = np.full((Q, N), np.nan)
        x[:, :: max(1, N // 9)] = rng.standard_normal((Q, len(range(0, N, max(1, N // 9)))))
        return x
    x = np.round(rng.standard_normal((Q, N)) * 2) / 2   # ties, +-0, infinities and NaN
    x[rng.random((Q, N)) < 0.05] = -0.0
    x[rng.random((Q, N)) < 0.001] = np.inf
    x[rng.random((Q, N)) < 0.01] = -np.inf
    x[rng.random((Q, N)) < 0.01] = np.nan
    return x


@pytest.mark.parametrize("kind", ["random", "descending", "blocks", "equal", "few", "mixed"])
@pytest.mark.parametrize("N,K", [(1, 1), (3, 5), (130, 20), (2047, 256), (4099, 20), (16384, 256), (16385, 20),
                                 (40_003, 256), (70_001, 1), (400_003, 256)])
def test_topk_select(N, K, kind):
    Q = 3
    rng = np.random.default_rng(N + K)
    x = rows(kind, Q, N, rng).astype(np.float32)
    # score[q][i] = <e_q, (x_0i, x_1i, x_2i)> would add 0 * NaN: rank each row on its own
    v, ix = O.top_k(x, K)
    for q in range(Q):
        tv, ti = E.score_topk(torch.from_numpy(x[q][:, None].copy()).to(DEV), None, [1], E.SCORE_FP,
                              torch.ones((1, 1), device=DEV), K)
        assert np.array_equal(ti.cpu().numpy()[0], ix[q])
        np.testing.assert_array_equal(tv.cpu().numpy()[0], v[q].astype(np.float32))
    E.sync_status()


def test_topk_select_many_queries():
    """Queries of one call: each row's slices and lists are its own."""
    rng = np.random.default_rng(5)
    x, y = rng.standard_normal((20_001, 8)).astype(np.float32), rng.standard_normal((37, 8)).astype(np.float32)
    tx, ty = torch.from_numpy(x).to(DEV), torch.from_numpy(y).to(DEV)
    v, ix = O.top_k(E.score(tx, None, [8], E.SCORE_FP, ty).cpu().numpy(), 30)
    tv, ti = E.score_topk(tx, None, [8], E.SCORE_FP, ty, 30)
    assert np.array_equal(ti.cpu().numpy(), ix)
    np.testing.assert_array_equal(tv.cpu().numpy(), v.astype(np.float32))
    E.sync_status()


def test_topk_rows_scored_in_chunks():
    """More scores than 1 GiB holds: rows are scored and ranked a chunk at a time."""
    N, Q, K = 300_001, 1000, 3
    gen = torch.Generator(device=DEV).manual_seed(3)
    x, y = torch.randn((N, 4), device=DEV, generator=gen), torch.randn((Q, 4), device=DEV, generator=gen)
    tv, ti = E.score_topk(x, None, [4], E.SCORE_FP, y, K)
    for q in (0, 511, 999):
        v, ix = O.top_k(E.score(x, None, [4], E.SCORE_FP, y[q:q + 1]).cpu().numpy(), K)
        assert np.array_equal(ti[q:q + 1].cpu().numpy(), ix)
        np.testing.assert_array_equal(tv[q:q + 1].cpu().numpy(), v.astype(np.float32))
    E.sync_status()
