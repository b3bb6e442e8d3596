"""The EK-FAC sums at the edges of their tiles: widths that leave ragged tiles of
either kernel, rows past the last pair, token counts around a K block, runs of
examples of unequal length, a strided destination and accumulation into it."""
import numpy as np
import pytest
import torch

from oracle import eogp_oracle as O
from paper_2609_37842_gb300 import eogp as E
from paper_2609_37842_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


# Fp32 sums of n products are off by at most gam(n) of the sum of the magnitudes (the
# probabilistic bound, lambda = 8, of roundings of 2^-23); a bf16 pair holds a value to
# 2^-18; the product of the two low halves, left out, is below 2^-18 of the whole.
def gam(n):
    return min(n, 8 * n ** 0.5) * 2.0 ** -23


@pytest.mark.parametrize("d_in,d_out,T,B", [(264, 520, 70, 3), (1000, 1368, 64, 2), (64, 2304, 130, 5), (1352, 72, 33, 4),
                                            (8, 8, 1, 1), (768, 3072, 65, 33), (136, 264, 63, 200), (320, 256, 129, 1)])
def test_ekfac_tiles(d_in, d_out, T, B):
    rng = np.random.default_rng(d_in * 7 + d_out + B)
    QA, QS = (synth.round_to(synth.haar_orthogonal(d, rng), "bf16") for d in (d_in, d_out))
    a = synth.round_to(rng.standard_normal((B, T, d_in)), "bf16")
    s = synth.round_to(rng.standard_normal((B, T, d_out)) * 0.1, "bf16")
    dv = lambda x: torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).to(DEV).to(torch.bfloat16)
    desc = E.ekfac_desc(T, dv(QA.T), dv(QS.T))
    A, S, VA, VS = (torch.from_numpy(np.asarray(x, dtype=np.float64)).to(DEV) for x in (a, s, QA, QS))
    want = torch.zeros((d_out, d_in), device=DEV, dtype=torch.float64)
    bar = torch.zeros_like(want)
    for b in range(B):
        at, st = A[b] @ VA, S[b] @ VS
        ea = 2.0 ** -18 * at.abs() + gam(d_in) * (A[b].abs() @ VA.abs())
        es = 2.0 ** -18 * st.abs() + gam(d_out) * (S[b].abs() @ VS.abs())
        g = st.T @ at
        e = st.abs().T @ ea + es.T @ (at.abs() + ea) + (2.0 ** -18 + gam(3 * T)) * (st.abs().T @ at.abs())
        want += g ** 2
        bar += (2 * g.abs() + e) * e + (g.abs() + e) ** 2 * gam(B)
    if d_in * d_out <= 200000 and B <= 5:
        assert np.allclose(want.cpu().numpy(), O.ekfac_sumsq(a, s, QA, QS), rtol=1e-9)
    one = E.ekfac_accumulate(desc, dv(a), dv(s))
    pad = torch.full((d_out, d_in + 3), 5.0, device=DEV, dtype=torch.float64)
    for n in range(2):
        E.ekfac_accumulate(desc, dv(a), dv(s), sumsq=pad[:, :d_in], accumulate=n > 0)
    E.sync_status()
    assert bool(((one - want).abs() <= bar).all())
    assert torch.equal(pad[:, :d_in], one + one) and bool((pad[:, d_in:] == 5.0).all())
