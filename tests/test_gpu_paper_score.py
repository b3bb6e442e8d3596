"""k_score_paper (unquantised queries, stored codes) at the edges of its tiles:
modules of odd numbers of 64-coordinate pairs and longer than an accumulation run,
query tiles of every width, ragged rows, several K ranges and (a workspace for the
queries alone) one, strided operands, and rows only the one-CTA kernel can read.
The bound is the documented 1e-5 sum_u s_iu ||y_qu||_1."""
import numpy as np
import pytest
import torch

from oracle import eogp_oracle as O
from paper_2609_37842_gb300 import eogp as E
from paper_2609_37842_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def padded(x, pad):
    t = torch.from_numpy(x.view(np.int32) if x.dtype == np.uint32 else x)
    base = torch.zeros((x.shape[0], x.shape[1] + pad), dtype=t.dtype, device=DEV)
    base[:, :x.shape[1]] = t.to(DEV)
    return base[:, :x.shape[1]]


@pytest.mark.parametrize("pad", [0, 4, 2])
@pytest.mark.parametrize("N,Q,ks", [(1, 1, [64]), (129, 16, [64, 1088, 128]), (200, 17, [1024] * 6), (300, 128, [2112]),
                                    (131, 129, [192, 64, 320]), (257, 250, [512, 1024, 64]), (1000, 33, [4096, 64])])
def test_paper_scores(N, Q, ks, pad):
    W = sum(k // 32 for k in ks)
    if pad == 0 and W % 4:
        pad = 4 - W % 4  # 16-byte rows
    tc = synth.random_codes(N, W, 31)
    ts = synth.lognormal_scales(N, len(ks), 0.5, 32)
    y = np.random.default_rng(Q).standard_normal((Q, sum(ks))).astype(np.float32)
    want = O.score_paper(tc, ts, ks, y)
    off = np.cumsum([0] + list(ks))
    bar = sum(np.abs(y[:, off[u]:off[u + 1]]).sum(1)[:, None] * ts[None, :, u] for u in range(len(ks))) * 1e-5
    a = (padded(tc, pad), padded(ts, 1), ks, E.SCORE_PAPER, padded(y, 3))
    out = torch.full((Q, N + 3), -7.0, device=DEV)
    E.score(*a, out=out[:, :N])
    one = E.score(*a, ws=torch.empty(-(-4 * Q * sum(ks) // 256) * 256, dtype=torch.uint8, device=DEV))
    E.sync_status()
    assert np.all(np.abs(out[:, :N].cpu().numpy() - want) <= bar)
    assert np.all(np.abs(one.cpu().numpy() - want) <= bar)
    assert bool((out[:, N:] == -7.0).all())
