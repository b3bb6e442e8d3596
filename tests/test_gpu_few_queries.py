"""One-bit scoring of fewer than 64 queries: the tensor-core path and the popcount
path (an empty workspace) against the oracle's float32 evaluation, bit for bit, on
both sides of every line of the dispatch (5, 9 and 17 queries; modules that are a
multiple of 256, of 128 or of nothing; rows the vector loads cannot take)."""
import numpy as np
import pytest
import torch

from oracle import eogp_oracle as O
from paper_2609_37842_gb300 import eogp as E
from paper_2609_37842_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def codes(n, ks, seed):
    W = sum((k + 31) // 32 for k in ks)
    c = synth.random_codes(n, W, seed)
    w = 0
    for k in ks:
        w += (k + 31) // 32
        if k % 32:
            c[:, w - 1] &= np.uint32((1 << (k % 32)) - 1)
    return c


def padded(x, pad):
    """x as a device view whose rows are `pad` elements apart from each other."""
    t = torch.from_numpy(x.view(np.int32) if x.dtype == np.uint32 else x)
    base = torch.zeros((x.shape[0], x.shape[1] + pad), dtype=t.dtype, device=DEV)
    base[:, :x.shape[1]] = t.to(DEV)
    return base[:, :x.shape[1]]


@pytest.mark.parametrize("Q", [1, 4, 5, 8, 9, 16, 17, 31, 33, 63])
@pytest.mark.parametrize("N,ks,pad", [(700, [4096], 0), (1, [16384], 4), (513, [1024], 0), (300, [1024] * 5, 8),
                                      (260, [256, 512, 256, 3328], 0), (257, [128, 640, 384], 4),
                                      (130, [1000, 96], 0), (300, [4096, 1024], 1)])
def test_few_query_codes_bit_exact(N, ks, pad, Q):
    tc, qc = codes(N, ks, 11), codes(Q, ks, 12)
    ts = synth.lognormal_scales(N, len(ks), 0.5, 13)
    qs = synth.lognormal_scales(Q, len(ks), 0.5, 14)
    want = O.score_codes_f32(tc, ts, ks, qc, qs)
    a = (padded(tc, pad), padded(ts, 0), ks, E.SCORE_CODES, padded(qc, pad), padded(qs, 3))
    out = torch.full((Q, N + 5), -7.0, device=DEV)
    got = E.score(*a, out=out[:, :N])
    assert np.array_equal(got.cpu().numpy(), want)
    assert bool((out[:, N:] == -7.0).all())
    pop = E.score(*a, ws=torch.empty(0, dtype=torch.uint8, device=DEV))
    assert np.array_equal(pop.cpu().numpy(), want)
    v, ix = O.top_k(want, min(7, N))
    tv, ti = E.score_topk(*a[:5], min(7, N), query_scales=a[5])
    assert np.array_equal(ti.cpu().numpy(), ix) and np.array_equal(tv.cpu().numpy(), v.astype(np.float32))
    E.sync_status()


def test_few_query_topk_of_unaligned_rows():
    """Rows the tensor cores cannot read are still ranked, beyond the size one block ranks too."""
    N, ks, Q = 50_001, [4096], 6
    tc, qc = codes(N, ks, 21), codes(Q, ks, 22)
    ts = synth.lognormal_scales(N, 1, 0.5, 23)
    qs = synth.lognormal_scales(Q, 1, 0.5, 24)
    v, ix = O.top_k(O.score_codes_f32(tc, ts, ks, qc, qs), 20)
    for pad in (0, 1):
        tv, ti = E.score_topk(padded(tc, pad), padded(ts, 0), ks, E.SCORE_CODES, padded(qc, 0), 20,
                              query_scales=padded(qs, 0))
        assert np.array_equal(ti.cpu().numpy(), ix) and np.array_equal(tv.cpu().numpy(), v.astype(np.float32))
    E.sync_status()
