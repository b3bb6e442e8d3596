"""What the performance of this framework is measured on: single calls of its public entry points, at the sizes its
workloads have (the five synthetic workloads of synth.py, the query and ranking workloads of bench.py) and between them.

A case is a dict of plain values; its "path" says which entry point runs:
  compress  eogp.compress_layer: one module's per-example gradients of a batch into codes (storing examples), coordinates
            (projecting queries) or first-stage coordinates (the rows the PCA is fitted on)
  ekfac     eogp.ekfac_accumulate: the EK-FAC eigenvalue correction of one module
  score     eogp.score: queries against stored examples, every score
  topk      eogp.score_topk: the best stored examples of every query
  fit       eogp.fit_pca: the one-time PCA fit of one module
"""
import math

import numpy as np
import torch

from paper_2609_37842_gb300 import eogp

DEV = "cuda"
OUT = {"first_stage": eogp.OUT_FIRST_STAGE, "coords": eogp.OUT_COORDS, "codes": eogp.OUT_CODES}
MODE = {"codes": eogp.SCORE_CODES, "paper": eogp.SCORE_PAPER, "fp": eogp.SCORE_FP}


def _compress(d_in, d_out, T, m, k, B, dtype="bf16", out="codes", spectrum="power", alpha=1.2, damping=0.1, a_std=1.0,
              s_std=0.1, stage2="pca", bias=False, ragged=False):
    return dict(path="compress", d_in=d_in, d_out=d_out, T=T, m=m, k=k, B=B, dtype=dtype, out=out, spectrum=spectrum,
                alpha=alpha, damping=damping, a_std=a_std, s_std=s_std, stage2=stage2, bias=bias, ragged=ragged)


def _ekfac(d_in, d_out, T, B, dtype="bf16", s_std=0.1):
    return dict(path="ekfac", d_in=d_in, d_out=d_out, T=T, B=B, dtype=dtype, a_std=1.0, s_std=s_std)


def _score(mode, N, Q, U, k, topk=0):
    c = dict(path="topk" if topk else "score", mode=mode, N=N, Q=Q, U=U, k=k)
    return dict(c, topk=topk) if topk else c


def _fit(n, m, k):
    return dict(path="fit", n=n, m=m, k=k)


def listed():
    return [
        # The fp32 layer of the smallest workload: its whole training set of 256 examples stored in one call (the smallest
        # call, where launches count), and a bulk store of 4096 examples.
        dict(_compress(64, 64, 16, 512, 128, 256, dtype="f32", alpha=1.5, damping=1e-3, s_std=1.0), name="store_f32_b256"),
        dict(_compress(64, 64, 16, 512, 128, 4096, dtype="f32", alpha=1.5, damping=1e-3, s_std=1.0), name="store_f32_b4096"),
        # A handful of interactive queries projected through a GPT-2 attention module: bias channel, texts of unequal
        # length padded to the block size; the coordinates stay unquantised (the query side of the paper's score).
        dict(_compress(768, 2304, 512, 4096, 1024, 5, out="coords", bias=True, ragged=True), name="query_gpt2_c_attn_b5"),
        # Storing a batch of training examples, module by module: the GPT-2 MLP input (short reductions, output-heavy),
        # the OLMo-2-7B gate (long reductions, the bulk of the largest workload) and the OLMo-2-1B down projection with
        # per-channel spectra and the SRHT second stage (few retained rows, bound by reading its inputs).
        dict(_compress(768, 3072, 512, 4096, 1024, 256, bias=True, ragged=True), name="store_gpt2_c_fc_b256"),
        dict(_compress(4096, 11008, 2048, 8192, 2048, 24, alpha=1.0), name="store_olmo7b_gate_b24"),
        dict(_compress(8192, 2048, 2048, 8192, 2048, 32, spectrum="channel", s_std=1.0, stage2="srht"), name="store_olmo1b_down_b32"),
        # The EK-FAC correction of a GPT-2 MLP module over a batch: once per module, before anything is stored.
        dict(_ekfac(768, 3072, 512, 32), name="ekfac_gpt2_c_fc_b32"),
        # The PCA fit of one module from cached first-stage rows: once per module.
        dict(_fit(4096, 2048, 512), name="fit_n4096_m2048_k512"),
        # A few one-bit queries scanned over a million stored 16,384-bit codes.
        dict(_score("codes", 1_000_000, 20, 1, 16384), name="scan_1m_q20"),
        # The GPT-2 query workload: 1024 one-bit queries ranked over 16,384 stored examples of 48 modules (top 20), a
        # smaller set of unquantised queries with every score, and the unquantised ablation on both sides.
        dict(_score("codes", 16384, 1024, 48, 1024, topk=20), name="topk_gpt2_q1024"),
        dict(_score("paper", 16384, 250, 48, 1024), name="paper_gpt2_q250"),
        dict(_score("fp", 16384, 48, 48, 1024), name="fp_gpt2_q48"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["f32", "query", "store", "store", "srht", "ekfac", "fit", "codes", "codes", "topk", "paper", "fp"])
    if kind == "f32":
        # small fp32 modules: any sizes
        d_in, d_out, T = _log(rng, 24, 160), _log(rng, 24, 160), _log(rng, 4, 64)
        m = rng.randint(min(64, d_in * d_out // 4), min(1024, d_in * d_out // 2))
        k = rng.randint(max(8, m // 8), max(9, m // 2))
        B = _log(rng, 1, max(2, min(4096, 65536 // T)))
        return _compress(d_in, d_out, T, m, k, B, dtype="f32", out=rng.choice(["codes", "codes", "coords", "first_stage"]),
                         alpha=1.5, damping=1e-3, s_std=1.0, bias=rng.random() < 0.3, ragged=rng.random() < 0.3)
    if kind == "query":
        # one to sixteen queries of any length through a module of GPT-2's or OLMo's size
        d_in, d_out = rng.choice([(768, 2304), (768, 768), (768, 3072), (3072, 768), (2048, 2048), (4096, 4096)])
        big = d_in + d_out > 4000
        m, k = (8192, 2048) if big else (4096, 1024)
        return _compress(d_in, d_out, _log(rng, 24, 2048 if big else 512), m, k, _log(rng, 1, 16), out=rng.choice(["coords", "codes"]),
                         alpha=1.0 if big else 1.2, bias=not big, ragged=True)
    if kind == "store":
        d_in, d_out = rng.choice([(768, 2304), (768, 768), (768, 3072), (3072, 768), (2048, 2048), (1600, 6400), (4096, 4096)])
        big = d_in + d_out > 4000
        T = _log(rng, 128, 2048 if big else 512)
        m = 8 * _log(rng, 256, 1024 if big else 512)
        k = m // 4 if rng.random() < 0.7 else rng.randint(m // 8, m // 4)
        B = max(1, min(256, _log(rng, 8, 65536 // T * 2)))
        return _compress(d_in, d_out, T, m, k, B, out=rng.choice(["codes", "codes", "codes", "first_stage"]),
                         alpha=rng.choice([1.0, 1.2]), bias=not big and rng.random() < 0.5, ragged=rng.random() < 0.5)
    if kind == "srht":
        d_in, d_out = rng.choice([(2048, 2048), (2048, 8192), (8192, 2048)])
        T = _log(rng, 256, 2048)
        m = 8 * rng.randint(256, 1024)
        return _compress(d_in, d_out, T, m, m // 4, max(1, min(64, _log(rng, 4, 65536 // T))), spectrum="channel", s_std=1.0,
                         stage2="srht", out=rng.choice(["codes", "codes", "coords"]), ragged=rng.random() < 0.5)
    if kind == "ekfac":
        d_in, d_out = rng.choice([(768, 2304), (768, 768), (768, 3072), (3072, 768), (2048, 2048), (1000, 1368)])
        T = _log(rng, 64, 1024)
        return _ekfac(d_in, d_out, T, max(1, _log(rng, 1, max(2, 16384 // T))))
    if kind == "fit":
        n, m = _log(rng, 200, 4096), _log(rng, 200, 2048)
        return _fit(n, m, rng.randint(min(n, m) // 8, min(n, m) // 4))
    if kind == "codes":
        # a scan over codes of one or several modules; the code widths of the workloads and some in between
        U = rng.choice([1, 1, 7, 48])
        k = rng.choice([1024, 2048, 4096, 8192, 16384]) if U == 1 else rng.choice([1024, 2048, 640, 1000])
        Q = _log(rng, 1, 1024)
        most = min(2_000_000, int(1.6e10 * 8 / (U * k * 8)), int(2e13 / (U * k * Q)))
        return _score("codes", _log(rng, min(5000, most // 2), most), Q, U, k)
    if kind == "topk":
        U = rng.choice([1, 12, 48])
        k = rng.choice([4096, 16384]) if U == 1 else 1024
        Q = _log(rng, 1, 1024)
        N = _log(rng, 3000, min(400_000, int(1.6e12 / (U * k * Q)) + 6000))
        return _score("codes", N, Q, U, k, topk=rng.choice([10, 20, 50]))
    if kind == "paper":
        U = rng.choice([1, 12, 48])
        k = rng.choice([2048, 4096]) if U == 1 else rng.choice([1024, 512])
        return _score("paper", _log(rng, 2000, 32768), _log(rng, 1, 250), U, k)
    U = rng.choice([1, 12, 48])
    return _score("fp", _log(rng, 1000, 16384), _log(rng, 1, 48), U, rng.choice([1024, 512, 1000]))


# ------------------------------------------------------------------ inputs
def _gen(seed, role):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1009 + role) & 0x7FFFFFFF)


def _dt(c):
    return torch.float32 if c["dtype"] == "f32" else torch.bfloat16


def _spectra(c, seed):
    """Factor spectra (d_out, then d_in with the bias channel), descending, and the channel scales they come from."""
    d_in = c["d_in"] + (1 if c["bias"] else 0)
    if c["spectrum"] == "power":
        return (np.arange(1, c["d_out"] + 1.0) ** -c["alpha"], np.arange(1, d_in + 1.0) ** -c["alpha"], None, None)
    r = np.random.default_rng(seed)
    ss = np.exp(r.uniform(math.log(0.1), math.log(10.0), c["d_out"]))
    sa = np.exp(r.uniform(math.log(0.1), math.log(10.0), d_in))
    return np.sort(ss ** 2)[::-1].copy(), np.sort(sa ** 2)[::-1].copy(), ss, sa


def _rows(d, n, seed, role):
    """n orthonormal rows of length d."""
    q, r = torch.linalg.qr(torch.randn((d, n), device=DEV, generator=_gen(seed, role)))
    s = torch.sign(torch.diagonal(r))
    s[s == 0] = 1.0
    return (q * s).t()


def _basis(d, idx, chan, seed, role):
    """The eigenvectors idx as rows: a random orthonormal basis, or the permutation that sorts the channels' scales."""
    if chan is None:
        return _rows(d, int(idx.max()) + 1, seed, role)[torch.as_tensor(idx, device=DEV).long()]
    cols = np.argsort(-chan ** 2, kind="stable")[np.asarray(idx)]
    v = torch.zeros((len(idx), d), device=DEV)
    v[torch.arange(len(idx), device=DEV), torch.as_tensor(cols.copy(), device=DEV)] = 1.0
    return v


def _tokens(c, d, std, chan, seed, role):
    """Activations or output gradients of a batch, B x T x d. An MLP's down projection (d_in > d_out) reads GELU outputs."""
    x = torch.randn((c["B"], c["T"], d), device=DEV, dtype=torch.float32 if c["dtype"] == "f32" else torch.bfloat16,
                    generator=_gen(seed, role))
    if role == 1 and c["d_in"] > c["d_out"] and c["dtype"] != "f32":
        x = torch.nn.functional.gelu(x)
    x *= std
    if chan is not None:
        x *= torch.as_tensor(chan[:d], device=DEV, dtype=x.dtype)
    return x


def _module(c, seed, R, C):
    """Everything a compression reads besides the plan: inputs, retained eigenvector rows, the second stage."""
    lam_S, lam_A, ss, sa = _spectra(c, seed)
    d_in = len(lam_A)
    VA = _basis(d_in, C, sa, seed, 3).to(_dt(c))
    VS = _basis(c["d_out"], R, ss, seed, 4).to(_dt(c)).contiguous()
    x = dict(a=_tokens(c, c["d_in"], c["a_std"], sa, seed, 1), s=_tokens(c, c["d_out"], c["s_std"], ss, seed, 2), VS=VS,
             VA=VA[:, :c["d_in"]].contiguous(), bias=VA[:, c["d_in"]].float().contiguous() if c["bias"] else None, lengths=None,
             Pt=None, signs=None, rows=None)
    if c["ragged"]:
        x["lengths"] = torch.randint(max(1, c["T"] // 8), c["T"] + 1, (c["B"],), device=DEV, dtype=torch.int32, generator=_gen(seed, 5))
    if c["out"] != "first_stage":
        if c["stage2"] == "pca":
            x["Pt"] = _rows(c["m"], c["k"], seed, 6).to(_dt(c)).contiguous()
        else:
            r = np.random.default_rng(seed + 1)
            p = 1 << (c["m"] - 1).bit_length()
            x["signs"] = torch.as_tensor(np.where(r.integers(0, 2, c["m"]) == 1, 1, -1).astype(np.int8), device=DEV)
            x["rows"] = torch.as_tensor(np.sort(r.choice(p, c["k"], replace=False)).astype(np.int32), device=DEV)
    return x


def _full_bases(c, seed):
    return (_rows(c["d_in"], c["d_in"], seed, 3).to(_dt(c)).contiguous(), _rows(c["d_out"], c["d_out"], seed, 4).to(_dt(c)).contiguous())


def _fit_rows(c, seed):
    """First-stage rows with a decaying spectrum in a mixed basis."""
    col = torch.arange(1, c["m"] + 1, device=DEV, dtype=torch.float32) ** -0.7
    return (torch.randn((c["n"], c["m"]), device=DEV, generator=_gen(seed, 1)) * col) @ _rows(c["m"], c["m"], seed, 2)


def _stored(c, seed):
    """Stored codes (or coordinates) and the queries, with their per-module scales."""
    D, W = c["U"] * c["k"], c["U"] * ((c["k"] + 31) // 32)

    def codes(n, role):
        x = torch.randint(-2 ** 31, 2 ** 31 - 1, (n, W), device=DEV, dtype=torch.int32, generator=_gen(seed, role))
        if c["k"] % 32:  # pad bits are zero
            last = torch.arange(1, c["U"] + 1, device=DEV) * ((c["k"] + 31) // 32) - 1
            x[:, last] &= (1 << (c["k"] % 32)) - 1
        return x

    def scales(n, role):
        return torch.exp(0.5 * torch.randn((n, c["U"]), device=DEV, generator=_gen(seed, role)))

    x = dict(ts=None, qs=None)
    if c["mode"] == "fp":
        x["train"] = torch.randn((c["N"], D), device=DEV, generator=_gen(seed, 1))
    else:
        x["train"], x["ts"] = codes(c["N"], 1), scales(c["N"], 2)
    if c["mode"] == "codes":
        x["query"], x["qs"] = codes(c["Q"], 3), scales(c["Q"], 4)
    else:
        x["query"] = torch.randn((c["Q"], D), device=DEV, generator=_gen(seed, 3))
    return x


def prepare(case, seed):
    c = case
    if c["path"] == "compress":
        lam_S, lam_A, _, _ = _spectra(c, seed)
        plan = eogp.Plan.from_factors(lam_S, lam_A, c["m"], c["damping"])
        x = _module(c, seed, *plan.sets())
        desc = eogp.layer_desc(plan, c["T"], c["k"], x["VA"], x["VS"], x["Pt"], srht_signs=x["signs"], srht_rows=x["rows"],
                               bias_A=x["bias"], lengths=x["lengths"])
        ws = eogp.workspace(eogp.compress_workspace_size(desc, c["B"], OUT[c["out"]]), DEV)
        return dict(path="compress", desc=desc, a=x["a"], s=x["s"], out=OUT[c["out"]], ws=ws)
    if c["path"] == "ekfac":
        VA, VS = _full_bases(c, seed)
        desc = eogp.ekfac_desc(c["T"], VA, VS)
        return dict(path="ekfac", desc=desc, a=_tokens(c, c["d_in"], c["a_std"], None, seed, 1), s=_tokens(c, c["d_out"], c["s_std"], None, seed, 2),
                    sumsq=torch.zeros((c["d_out"], c["d_in"]), device=DEV, dtype=torch.float64),
                    ws=eogp.workspace(eogp.ekfac_workspace_size(desc, c["B"]), DEV))
    if c["path"] == "fit":
        return dict(path="fit", Z=_fit_rows(c, seed), k=c["k"], ws=eogp.workspace(eogp.fit_pca_workspace_size(c["n"], c["m"], c["k"]), DEV))
    return dict(_stored(c, seed), path=c["path"], ks=[c["k"]] * c["U"], mode=MODE[c["mode"]], topk=c.get("topk"))


def run(state):
    x = state
    if x["path"] == "compress":
        return eogp.compress_layer(x["desc"], x["a"], x["s"], x["out"], ws=x["ws"])
    if x["path"] == "ekfac":
        return eogp.ekfac_accumulate(x["desc"], x["a"], x["s"], sumsq=x["sumsq"], ws=x["ws"])
    if x["path"] == "fit":
        return eogp.fit_pca(x["Z"], x["k"], ws=x["ws"])
    if x["path"] == "topk":
        return eogp.score_topk(x["train"], x["ts"], x["ks"], x["mode"], x["query"], x["topk"], query_scales=x["qs"])
    return eogp.score(x["train"], x["ts"], x["ks"], x["mode"], x["query"], query_scales=x["qs"])


# ------------------------------------------------------------------ work
def _sets(c, seed=0):
    """Retained rows and columns (R, C), the retained coordinates (j, i) in their order and their scales, in 64 bits: the m
    largest products of the two spectra, ties to the lower Kronecker position i * d_out + j."""
    lam_S, lam_A, _, _ = _spectra(c, seed)
    v = (lam_A[:, None] * lam_S[None, :]).reshape(-1)
    lam = c["damping"] * v.sum() / v.size
    t = np.partition(v, v.size - c["m"])[v.size - c["m"]]
    pos = np.flatnonzero(v >= t)
    pos = pos[np.argsort(-v[pos], kind="stable")][:c["m"]]
    i, j = pos // len(lam_S), pos % len(lam_S)
    return np.unique(j), np.unique(i), j, i, 1.0 / np.sqrt(v[pos] + lam)


def work(case):
    c = case
    if c["path"] == "compress":
        R, C, _, _, _ = _sets(c)
        e = 4 if c["dtype"] == "f32" else 2
        M = c["B"] * c["T"]
        outs = {"first_stage": 4 * c["m"], "coords": 4 * c["k"], "codes": c["k"] / 8 + 4}[c["out"]]
        b = e * M * (c["d_in"] + c["d_out"]) + e * (len(R) * c["d_out"] + len(C) * c["d_in"]) + c["B"] * outs
        f = 2 * M * (c["d_in"] * len(C) + c["d_out"] * len(R)) + 2 * M * c["m"]
        if c["out"] != "first_stage":
            b += e * c["k"] * c["m"] if c["stage2"] == "pca" else c["m"] + 4 * c["k"]
            f += c["B"] * (2 * c["m"] * c["k"] if c["stage2"] == "pca" else c["m"] * math.log2(c["m"]))
        return {"bytes": b, "flops": f}
    if c["path"] == "ekfac":
        e, M = (4 if c["dtype"] == "f32" else 2), c["B"] * c["T"]
        return {"bytes": e * (M * (c["d_in"] + c["d_out"]) + c["d_in"] ** 2 + c["d_out"] ** 2) + 8 * c["d_in"] * c["d_out"],
                "flops": 2 * M * (c["d_in"] ** 2 + c["d_out"] ** 2 + c["d_in"] * c["d_out"])}
    if c["path"] == "fit":
        n, m, k, nn = c["n"], c["m"], c["k"], min(c["n"], c["m"])
        # one half of the symmetric second moment, one product of it with k vectors and their orthonormalisation
        return {"bytes": 4 * (n * m + k * m + k), "flops": nn * nn * max(n, m) + 2 * nn * nn * k + 2 * nn * k * k}
    D, W = c["U"] * c["k"], c["U"] * ((c["k"] + 31) // 32)
    per = 4 * D if c["mode"] == "fp" else 4 * W + 4 * c["U"]
    query = 4 * W + 4 * c["U"] if c["mode"] == "codes" else 4 * D
    outs = 8 * c["topk"] if c["path"] == "topk" else 4 * c["N"]
    return {"bytes": c["N"] * per + c["Q"] * (query + outs), "flops": 2 * c["N"] * c["Q"] * D}


# ------------------------------------------------------------------ the same in 64 bits
def _exact_compress(c, seed):
    R, C, j, i, scale = _sets(c, seed)
    x = _module(c, seed, R, C)
    VA, VS, scale = x["VA"].double(), x["VS"].double(), torch.as_tensor(scale, device=DEV)
    jr = torch.as_tensor(np.searchsorted(R, j), device=DEV)
    ic = torch.as_tensor(np.searchsorted(C, i), device=DEV)
    z = torch.empty((c["B"], c["m"]), device=DEV, dtype=torch.float64)
    step = max(1, min(c["B"], 16384 // c["T"]))
    for b in range(0, c["B"], step):
        at = x["a"][b:b + step].double() @ VA.t()
        st = x["s"][b:b + step].double() @ VS.t()
        if x["bias"] is not None:
            at += x["bias"].double()
        if x["lengths"] is not None:
            st *= (torch.arange(c["T"], device=DEV)[None, :] < x["lengths"][b:b + step, None])[:, :, None]
        z[b:b + step] = (st.transpose(1, 2) @ at)[:, jr, ic] * scale
    if c["out"] == "first_stage":
        return z
    if c["stage2"] == "pca":
        y = z @ x["Pt"].double().t()
    else:
        p = 1 << (c["m"] - 1).bit_length()
        y = torch.zeros((c["B"], p), device=DEV, dtype=torch.float64)
        y[:, :c["m"]] = z * x["signs"].double()
        h = 1
        while h < p:
            w = y.view(c["B"], p // (2 * h), 2, h)
            y = torch.stack((w[:, :, 0] + w[:, :, 1], w[:, :, 0] - w[:, :, 1]), 2).reshape(c["B"], p)
            h *= 2
        y = y[:, x["rows"].long()] / math.sqrt(c["k"])
    return y if c["out"] == "coords" else (None, y.abs().mean(1))


def _signs(words, U, k):
    """+-1 per stored coordinate, in 64 bits."""
    b = torch.arange(32, device=DEV, dtype=torch.int32)
    x = ((words[:, :, None] >> b) & 1).reshape(words.shape[0], U, -1)[:, :, :k]
    return (2 * x - 1).double()


def _exact_score(c, seed):
    x = _stored(c, seed)
    if c["mode"] == "fp":
        q = x["query"].double()
    elif c["mode"] == "paper":
        q = x["query"].double()
    else:
        q = (_signs(x["query"], c["U"], c["k"]) * x["qs"].double()[:, :, None]).reshape(c["Q"], -1)
    out = torch.empty((c["Q"], c["N"]), device=DEV, dtype=torch.float64)
    step = max(1, min(c["N"], (1 << 28) // (c["U"] * c["k"])))
    for r in range(0, c["N"], step):
        t = x["train"][r:r + step]
        if c["mode"] == "fp":
            t = t.double()
        else:
            t = (_signs(t, c["U"], c["k"]) * x["ts"][r:r + step].double()[:, :, None]).reshape(t.shape[0], -1)
        out[:, r:r + step] = q @ t.t()
    return out if c["path"] == "score" else (torch.topk(out, c["topk"], dim=1).values, None)


def exact(case, seed):
    c = case
    if c["path"] == "compress":
        return _exact_compress(c, seed)
    if c["path"] == "ekfac":
        VA, VS = _full_bases(c, seed)
        at = _tokens(c, c["d_in"], c["a_std"], None, seed, 1).double() @ VA.double().t()
        st = _tokens(c, c["d_out"], c["s_std"], None, seed, 2).double() @ VS.double().t()
        out = torch.zeros((c["d_out"], c["d_in"]), device=DEV, dtype=torch.float64)
        for b in range(c["B"]):
            out += (st[b].t() @ at[b]).square()
        return out
    if c["path"] == "fit":
        Z = _fit_rows(c, seed).double()
        gram = c["n"] < c["m"]
        w, v = torch.linalg.eigh((Z @ Z.t() if gram else Z.t() @ Z) / c["n"])
        w, v = w.flip(0)[:c["k"]], v.flip(1)[:, :c["k"]]
        # directions of the large fits are returned at a residual of 1e-3 of their eigenvalue: among close eigenvalues that
        # leaves them no single value
        if min(c["n"], c["m"]) > 1024:
            return None, w
        P = (Z.t() @ v if gram else v).t()
        P = P / P.norm(dim=1, keepdim=True)
        at = P.abs().argmax(1, keepdim=True)
        return P * torch.sign(torch.gather(P, 1, at)), w
    return _exact_score(c, seed)
