"""Calls from several host threads at once, each with a module of its own size: the
limit of a kernel's dynamic shared memory belongs to the process, so one thread's
smaller need must not refuse another's launch. The calls go straight to the library,
which leaves the interpreter lock, often enough to meet in the short time between."""
import ctypes
import threading

import pytest
import torch

from paper_2609_37842_gb300 import eogp as E
from paper_2609_37842_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


class Module:
    def __init__(self, d_in, d_out, T, m, k, B, dtype, seed, srht=False):
        g = torch.Generator(DEV).manual_seed(seed)
        plan = E.Plan.from_factors(synth.power_spectrum(d_out, 1.1), synth.power_spectrum(d_in, 1.2), m, 0.1)
        R, C = plan.sets()
        rnd = lambda *s: torch.randn(s, device=DEV, generator=g).to(dtype)
        second = dict(srht_signs=torch.ones(m, dtype=torch.int8, device=DEV),
                      srht_rows=torch.arange(k, dtype=torch.int32, device=DEV)) if srht else {}
        VA, VS, Pt = rnd(len(C), d_in), rnd(len(R), d_out), None if srht else rnd(k, m)
        desc = E.layer_desc(plan, T, k, VA, VS, Pt, **second)
        ws = E.workspace(E.compress_workspace_size(desc, B, E.OUT_COORDS), DEV)
        a, s = rnd(B, T, d_in), rnd(B, T, d_out)
        self.out, self.stream = torch.zeros((B, k), device=DEV), torch.cuda.Stream()
        self.keep = plan, second, VA, VS, Pt, desc, ws, a, s
        self.want = E.compress_layer(desc, a, s, E.OUT_COORDS, ws=ws)
        self.args = (ctypes.byref(desc), E._ptr(a), E._ptr(s), B, E.OUT_COORDS, E._ptr(self.out), self.out.stride(0), None, 0,
                     None, 0, E._ptr(ws), ws.numel(), self.stream.cuda_stream)

    def call(self):
        return E.lib().eogp_compress_layer(*self.args)


F, H = torch.float32, torch.bfloat16
KINDS = {
    "fp32": [(64, 64, 30, 512, 128, 8, F, 1), (200, 120, 30, 4000, 64, 8, F, 2), (24, 32, 30, 60, 16, 8, F, 3)],
    "bf16": [(256, 384, 128, 1024, 256, 4, H, 4), (768, 512, 64, 4096, 256, 2, H, 5)],
    "srht": [(128, 128, 16, 256, 64, 4, H, 7, True), (512, 512, 16, 8192, 64, 4, H, 8, True)],
}


@pytest.mark.parametrize("kind", KINDS)
def test_threads(kind):
    modules = [Module(*a) for a in KINDS[kind]]
    torch.cuda.synchronize()
    start, refused = threading.Barrier(len(modules)), [0] * len(modules)

    def work(i):
        start.wait()
        for n in range(20000):
            refused[i] += modules[i].call() != 0
            if n % 500 == 0:
                modules[i].stream.synchronize()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(modules))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    E.sync_status()
    assert refused == [0] * len(modules)
    for m in modules:
        assert torch.equal(m.out, m.want)
