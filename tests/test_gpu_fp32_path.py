"""The fp32 kernels at the edges of their tiles: k_f32_first against the oracle
(one and several examples per block, token counts that do and do not vectorise,
ragged columns, bias and lengths, modules just past what it takes), k_simt_gemm
through the projection, and the tensor-core FP scores, infinities and NaN included."""
import numpy as np
import pytest
import torch

from oracle import eogp_oracle as O
from paper_2609_37842_gb300 import eogp as E
from paper_2609_37842_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def dt(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


@pytest.mark.parametrize("bias,ragged", [(False, False), (True, True)])
@pytest.mark.parametrize("d_in,d_out,T,m,k,B", [(64, 64, 16, 512, 128, 9), (33, 70, 1, 100, 31, 65), (65, 40, 5, 300, 64, 3),
                                                (24, 160, 16, 1000, 500, 2), (64, 64, 16, 512, 128, 700),
                                                (130, 129, 64, 777, 100, 3), (48, 50, 63, 200, 40, 5),
                                                (48, 50, 65, 200, 40, 4), (500, 300, 33, 2000, 130, 3)])
def test_fp32_compress(d_in, d_out, T, m, k, B, bias, ragged):
    rng = np.random.default_rng(d_in * 31 + B)
    di = d_in + (1 if bias else 0)
    QA, QS = (synth.haar_orthogonal(d, rng).astype(np.float32) for d in (di, d_out))
    lam_A, lam_S = synth.power_spectrum(di, 1.3), synth.power_spectrum(d_out, 1.1)
    plan = E.Plan.from_factors(lam_S, lam_A, m, 1e-2)
    R, C = plan.sets()
    j, i, scale = plan.retained()
    a, s = rng.standard_normal((B, T, d_in)).astype(np.float32), rng.standard_normal((B, T, d_out)).astype(np.float32)
    P = synth.haar_orthogonal(m, rng, k).astype(np.float32)
    lengths = rng.integers(0, T + 1, B).astype(np.int32) if ragged else None
    VA = QA[:d_in, C].T
    desc = E.layer_desc(plan, T, k, dt(VA), dt(QS[:, R].T), dt(P.T), bias_A=dt(QA[d_in, C]) if bias else None,
                        lengths=dt(lengths) if ragged else None)
    ta, ts = dt(a), dt(s)
    z = E.compress_layer(desc, ta, ts, E.OUT_FIRST_STAGE).cpu().numpy()
    x = E.compress_layer(desc, ta, ts, E.OUT_COORDS).cpu().numpy()
    codes, sc = E.compress_layer(desc, ta, ts, E.OUT_CODES)
    E.sync_status()
    at = a.astype(np.float64) @ QA[:d_in].astype(np.float64)
    if bias:
        at += QA[d_in].astype(np.float64)
    st = s.astype(np.float64) @ QS.astype(np.float64)
    if ragged:
        st *= (np.arange(T)[None, :] < lengths[:, None])[:, :, None]
    g = np.einsum("btj,bti->bji", st, at)
    want = g[:, j, i] * scale.astype(np.float64)
    bar = 1e-5 * np.linalg.norm(want, axis=1) + 1e-30
    assert np.all(np.linalg.norm(z - want, axis=1) <= bar)
    wx = want @ P.astype(np.float64)
    assert np.all(np.linalg.norm(x - wx, axis=1) <= 1e-5 * np.linalg.norm(wx, axis=1) + 1e-30)
    bits = np.unpackbits(codes.cpu().numpy().view(np.uint8), axis=1, bitorder="little")[:, :k].astype(bool)
    assert np.array_equal(bits, x >= 0)
    np.testing.assert_allclose(sc.cpu().numpy(), np.abs(x).mean(1), rtol=1e-5)


# |error| of an fp32 sum of D products taken in any order is at most D 2^-24 of
# the sum of their magnitudes; the split leaves out less than 2^-22 of it.
def fp_bar(x, y):
    return (x.shape[1] * 2.0 ** -24 + 2.0 ** -22) * (np.abs(y).astype(np.float64) @ np.abs(x).astype(np.float64).T)


@pytest.mark.parametrize("N,Q,D", [(1, 1, 256), (130, 3, 300), (129, 16, 1000), (257, 17, 512), (300, 48, 2049),
                                   (700, 64, 777), (128, 65, 4096), (1000, 150, 289), (3000, 5, 12288), (90, 2, 255)])
def test_fp_scores(N, Q, D):
    rng = np.random.default_rng(N + Q + D)
    x = (rng.standard_normal((N, D)) * np.exp(rng.uniform(-20, 20, (N, 1)))).astype(np.float32)
    y = (rng.standard_normal((Q, D)) * np.exp(rng.uniform(-20, 20, (Q, 1)))).astype(np.float32)
    pad = torch.zeros((N, (D + 3) // 4 * 4 + 4), device=DEV)
    pad[:, :D] = dt(x)
    out = torch.full((Q, N + 3), -7.0, device=DEV)
    E.score(pad[:, :D], None, [D], E.SCORE_FP, dt(y), out=out[:, :N])
    E.sync_status()
    got = out[:, :N].cpu().numpy()
    assert np.all(np.abs(got - O.score_fp(x, y)) <= fp_bar(x, y))
    assert bool((out[:, N:] == -7.0).all())
    # the CUDA-core kernel (no workspace) agrees to the same bound
    cc = E.score(pad[:, :D], None, [D], E.SCORE_FP, dt(y), ws=torch.empty(0, dtype=torch.uint8, device=DEV))
    assert np.all(np.abs(got - cc.cpu().numpy()) <= 2 * fp_bar(x, y))


def test_fp_scores_infinities_and_nan():
    """Rows and queries with an infinity or NaN give what IEEE fp32 sums give."""
    rng = np.random.default_rng(1)
    N, Q, D = 600, 70, 512
    x, y = (rng.integers(-4, 5, (n, D)).astype(np.float32) for n in (N, Q))
    x[5, 7], x[300, 0], x[301, 3], x[301, 4] = np.inf, np.nan, np.inf, -np.inf
    y[2, 100], y[69, 5] = -np.inf, np.nan
    x[17, 2] = np.finfo(np.float32).max
    # the fp32 sum, one rounding per step (a double holds every product here exactly):
    # what overflows in fp32 is infinite in it, as it is not in a 64-bit sum
    want = np.zeros((Q, N), np.float32)
    with np.errstate(all="ignore"):
        for c in range(D):
            want = (want.astype(np.float64) + y[:, c, None].astype(np.float64) * x[None, :, c]).astype(np.float32)
    got = E.score(dt(x), None, [D], E.SCORE_FP, dt(y))
    E.sync_status()
    got = got.cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(np.isposinf(got), np.isposinf(want)) and np.array_equal(np.isneginf(got), np.isneginf(want))
    small = np.isfinite(want) & (np.abs(want) < 2 ** 24)
    assert np.array_equal(got[small], want[small])


def test_fp_topk_beyond_one_chunk_of_k():
    rng = np.random.default_rng(2)
    x, y = rng.standard_normal((5000, 1024)).astype(np.float32), rng.standard_normal((9, 1024)).astype(np.float32)
    v, ix = O.top_k(E.score(dt(x), None, [512, 512], E.SCORE_FP, dt(y)).cpu().numpy(), 20)
    tv, ti = E.score_topk(dt(x), None, [512, 512], E.SCORE_FP, dt(y), 20)
    E.sync_status()
    assert np.array_equal(ti.cpu().numpy(), ix)
    np.testing.assert_array_equal(tv.cpu().numpy(), v.astype(np.float32))
