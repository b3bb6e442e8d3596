"""Both rotations of a module in one launch (few token rows) against the two launches
of a larger batch, at the edges of their tiles: widths that leave ragged tiles and
tiles past the padded width, token counts that are no multiple of 128, bias and
lengths; and the chain of dependent launches replayed from a captured graph."""
import numpy as np
import pytest
import torch

from paper_2609_37842_gb300 import eogp as E
from paper_2609_37842_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def case(dtype, d_in, d_out, T, m, k, B, bias, seed):
    rng = np.random.default_rng(seed)
    rnd = lambda v: synth.round_to(v, dtype)
    QA = rnd(synth.haar_orthogonal(d_in + (1 if bias else 0), rng))
    QS = rnd(synth.haar_orthogonal(d_out, rng))
    plan = E.Plan.from_factors(synth.power_spectrum(d_out, 1.1), synth.power_spectrum(QA.shape[0], 1.1), m, 1e-2)
    R, C = plan.sets()
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    dv = lambda x: torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).to(DEV).to(tdt)
    Pt = dv(rnd(synth.haar_orthogonal(m, rng, k).T))
    b = torch.from_numpy(np.ascontiguousarray(QA[d_in, C], dtype=np.float32)).to(DEV) if bias else None
    gen = torch.Generator(DEV).manual_seed(seed)
    a = torch.randn((B, T, d_in), device=DEV, generator=gen).to(tdt)
    s = (torch.randn((B, T, d_out), device=DEV, generator=gen) * 0.1).to(tdt)
    lens = torch.from_numpy(rng.integers(0, T + 1, B).astype(np.int32)).to(DEV) if bias else None
    desc = lambda n: E.layer_desc(plan, T, k, dv(QA[:d_in, C].T), dv(QS[:, R].T), Pt, bias_A=b, lengths=n)
    return plan, QA, QS, desc, a, s, b, lens


# The order of every sum is that of the K blocks, whatever tile and launch hold it, so
# the results are equal bit for bit; those of the larger batch are compared with the
# oracle elsewhere.
@pytest.mark.parametrize("d_in,d_out,T,m,B,bias", [(768, 768, 128, 2000, 70, False), (200, 136, 100, 704, 220, True),
                                                   (768, 2304, 96, 4096, 70, True), (1368, 1000, 50, 3000, 140, False),
                                                   (40, 1352, 64, 504, 260, True), (136, 72, 1, 304, 21000, False)])
def test_rotations_in_one_launch(d_in, d_out, T, m, B, bias):
    *_, desc, a, s, _, lens = case("bf16", d_in, d_out, T, m, 64, B, bias, d_in + d_out)
    z = E.compress_layer(desc(lens), a, s, E.OUT_FIRST_STAGE)
    for lo, hi in ((0, 1), (1, 4), (B - 2, B)):
        n = lens[lo:hi].clone() if bias else None
        got = E.compress_layer(desc(n), a[lo:hi].clone(), s[lo:hi].clone(), E.OUT_FIRST_STAGE)
        E.sync_status()
        assert torch.equal(got, z[lo:hi])


@pytest.mark.parametrize("dtype,d_in,d_out,T,m,k,B", [("bf16", 768, 768, 100, 2000, 300, 3), ("bf16", 200, 136, 64, 704, 64, 300),
                                                      ("f32", 64, 64, 16, 512, 128, 100), ("f32", 64, 64, 16, 512, 128, 1000)])
def test_captured_chain(dtype, d_in, d_out, T, m, k, B):
    *_, desc, a, s, _, _ = case(dtype, d_in, d_out, T, m, k, B, False, B)
    d = desc(None)
    ws = E.workspace(max(E.compress_workspace_size(d, B, o) for o in (E.OUT_CODES, E.OUT_COORDS)), DEV)
    want = [E.compress_layer(d, a, s, E.OUT_COORDS, ws=ws), *E.compress_layer(d, a, s, E.OUT_CODES, ws=ws)]
    a2, s2 = torch.zeros_like(a), torch.zeros_like(s)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        got = [E.compress_layer(d, a2, s2, E.OUT_COORDS, ws=ws), *E.compress_layer(d, a2, s2, E.OUT_CODES, ws=ws)]
    a2.copy_(a)
    s2.copy_(s)
    for _ in range(2):
        g.replay()
    E.sync_status()
    assert all(torch.equal(x, y) for x, y in zip(want, got))
