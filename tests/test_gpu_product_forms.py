"""The forms that a context's dot products run in (key MAC, BConv, fixed tensor
shapes): sums on limbs where every prime is below 2^60, 128-bit sums otherwise,
and in either case the reduction for primes = 1 (mod 2^32) where all are and
"q1_forms" is on. Read off the names of the kernels that a product, a wave and
a tensor product launch; the residues are the oracle's in every form."""
import re

import numpy as np
import pytest

import synth
from oracle import ckks as O

from gpu_common import Setup, dev, host, oracle_tuple

pytestmark = pytest.mark.gpu

K_IN = 4
# (q1, limb) of a kernel by its template arguments
FORM = [re.compile(r"\bbconv(?:_table)?_kernel<\d+, (\w+), (\w+)>"),
        re.compile(r"\bmac(?:_table)?_kernel<(\w+), \d+, \d+, (\w+)>"),
        re.compile(r"\btensor_fixed(?:_table)?_kernel<\d+, \d+, \d+, \d+, (\w+), (\w+)>")]


def _forms(call):
    """The forms of the kernels that call() launches, per kernel family."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    for _ in range(3):  # a process's first profile can come back without any kernel
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            call()
            torch.cuda.synchronize()
        names = {e.name for e in p.events()}
        if any("ckks" in n for n in names):
            break
    return [{tuple(x in ("true", "1") for x in m.groups()) for m in map(r.search, names) if m} for r in FORM]


@pytest.mark.parametrize("bits,limb", [([61, 50, 50], False), ([50, 50, 50], True)])
@pytest.mark.parametrize("congruence", [synth.Q1_CONGRUENCE, synth.NTT_CONGRUENCE])
def test_kernels_run_in_the_form_of_the_primes(bits, limb, congruence):
    import paper_2601_15401_gb300 as G
    p = synth.make_params(10, bits, 1, 3, congruence=congruence)
    S = Setup(p, K_IN, 960)
    cts = [synth.uniform_tuple(p, 2, p.L, 960, i) for i in range(K_IN)]
    want = O.mul_k(S.octx, [oracle_tuple(c) for c in cts], S.okeys).data
    ins = [S.tuple(c) for c in cts]
    out = S.tuple(np.zeros(want.shape, np.uint64))
    wave_out = S.tuple(np.zeros(want.shape, np.uint64))
    ws = S.ws(S.ctx.workspace_size(K_IN, p.L))
    wave = G.Wave(S.ctx, [(ins, wave_out, None)], S.evk)
    buffers = wave.buffers()
    g = synth.rng(961)
    fours = [np.stack([synth.uniform_residues(g, p.q, p.N) for _ in range(4)]) for _ in range(2)]
    prod = G.Tuple.wrap(dev(np.zeros((7, p.L, p.N), np.uint64)))

    def call():
        S.ctx.mul_k(ins, S.evk, out, ws)
        wave.run(*buffers)
        S.ctx.tensor([S.tuple(f) for f in fours], prod)

    for on in (1, 0):
        S.ctx.tune_set("q1_forms", on)
        call()
        q1 = bool(on) and congruence == synth.Q1_CONGRUENCE
        assert _forms(call) == [{(q1, limb)}] * len(FORM)
        S.ctx.check()
        assert np.array_equal(host(out.data), want)
        assert np.array_equal(host(wave_out.data), want)
        assert np.array_equal(host(prod.data), O.tensor_product(S.octx, fours))
