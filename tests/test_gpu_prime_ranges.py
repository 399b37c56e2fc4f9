"""Residues at the edges of the kernels' ranges, against the oracle.

The transforms choose their form by the size of each prime (below 2^53, below
2^60, below 2^61) and by the ring degree (run-time modes up to N = 2^8, one
launch up to 2^12, two phases above); dot products run on limbs when every
prime is below 2^60 and as 128-bit products otherwise, BConv in chunks of
eight sources, the key MAC with or without folding, ModUp transforms with as
many digits per launch as fit, and the NTT-domain ModDown through its own
conversion kernel when the buffers allow. Every comparison is bit for bit."""
import numpy as np
import pytest

import synth
from oracle import ckks as O
from oracle import ring as R

from gpu_common import Setup, dev, host, oracle_tuple

pytestmark = pytest.mark.gpu

# one prime on each side of every size bound, P primes of 60 bits
SIZES = [45, 52, 53, 54, 59, 60, 61]


@pytest.mark.parametrize("log_n", range(4, 17))
def test_transforms_of_every_prime_size(log_n):
    import paper_2601_15401_gb300 as G
    p = synth.make_params(log_n, SIZES, 2, 7)
    ctx = G.Context.from_params(p)
    g = synth.rng(77, log_n)
    x = np.stack([synth.uniform_residues(g, p.q, p.N), np.zeros((p.L, p.N), np.uint64),
                  np.stack([np.full(p.N, q - 1, np.uint64) for q in p.q]),
                  np.stack([np.where(np.arange(p.N) % 2 == 0, np.uint64(q - 1), np.uint64(0)) for q in p.q])])
    t = G.Tuple(dev(x), len(x), p.L, p.L, 0)
    f = G.Tuple(dev(np.zeros_like(x)), len(x), p.L, p.L, 0)
    ctx.ntt(t, f)
    assert np.array_equal(host(f.data), np.stack([R.ntt_rows(a, p.q) for a in x]))
    t = G.Tuple(dev(x), len(x), p.L, p.L, 1)
    ctx.intt(t, f)
    ctx.check()
    assert np.array_equal(host(f.data), np.stack([R.intt_rows(a, p.q) for a in x]))


# (log N, bits of q, special primes, dnum, k): digits of 2, 5, 12 and 16
# primes, one prime per digit (more limbs than one launch lists), primes of 60
# bits (wide sums, folded keys) and of 61 (128-bit products)
PRODUCTS = [
    (10, [45, 61, 50, 53, 60, 54], 3, 3, 3),
    (10, [60] * 6, 4, 3, 5),
    (9, [50] * 10, 5, 2, 4),
    (11, [50] * 12, 12, 1, 3),
    (10, [45] * 16, 6, 1, 4),
    (10, [50] * 12, 4, 12, 5),
    (13, [61] + [50] * 4, 2, 5, 4),
    (13, [60, 52, 53, 54, 45], 3, 2, 3),
]


@pytest.mark.parametrize("case", range(len(PRODUCTS)))
def test_products_over_digit_and_prime_ranges(case):
    import paper_2601_15401_gb300 as G
    log_n, bits, K, dnum, k = PRODUCTS[case]
    p = synth.make_params(log_n, bits, K, dnum)
    S = Setup(p, k, 900 + case)
    cts = [synth.uniform_tuple(p, 2, p.L, 900 + case, i) for i in range(k)]
    want = O.mul_k(S.octx, [oracle_tuple(c) for c in cts], S.okeys).data
    depth = S.ctx.plan_describe(k)["depth"]
    ws = S.ws(S.ctx.workspace_size(k, p.L))
    for fixed in (1, 0):
        S.ctx.tune_set("tensor_fixed", fixed)
        out = S.tuple(np.zeros((2, p.L - depth, p.N), np.uint64))
        S.ctx.mul_k([S.tuple(c) for c in cts], S.evk, out, ws)
        assert np.array_equal(host(out.data), want), fixed
    # the same product in a wave, beside a two-input one
    items = [([S.tuple(c) for c in cts], S.tuple(np.zeros((2, p.L - depth, p.N), np.uint64)), None),
             ([S.tuple(c) for c in cts[:2]], S.tuple(np.zeros((2, p.L - 1, p.N), np.uint64)), None)]
    w = G.Wave(S.ctx, items, S.evk)
    w.run(*w.buffers())
    S.ctx.check()
    assert np.array_equal(host(items[0][1].data), want)
    assert np.array_equal(host(items[1][1].data), O.mul_k(S.octx, [oracle_tuple(c) for c in cts[:2]], S.okeys).data)


# NTT-domain ModDown: K on both sides of the conversion kernel's chunk of
# eight and of its largest K, and a buffer too small for it (one digit, K < level)
@pytest.mark.parametrize("bits,K,dnum", [([50] * 4, 1, 1), ([50] * 4, 1, 2), ([50] * 6, 9, 2), ([60, 45, 53], 16, 1),
                                         ([50] * 3, 17, 1), ([61, 50, 50], 2, 3)])
@pytest.mark.parametrize("log_n", [10, 13])
def test_two_input_product_over_special_primes(log_n, bits, K, dnum):
    # more than 15 P primes of 60 bits would sum to 2^64 or more
    p = synth.make_params(log_n, bits, K, dnum, p_bits=60 if K <= 15 else 59)
    S = Setup(p, 2, 950 + K)
    a, b = (synth.uniform_tuple(p, 2, p.L, 950, i) for i in range(2))
    out = S.tuple(np.zeros((2, p.L - 1, p.N), np.uint64))
    S.ctx.mul2(S.tuple(a), S.tuple(b), S.evk, out, S.ws(S.ctx.mul2_workspace_size(p.L)))
    S.ctx.check()
    assert np.array_equal(host(out.data), O.mul2_standard(S.octx, oracle_tuple(a), oracle_tuple(b), S.okeys).data)


# signed loads: values on both sides of the fast path's bound (2^61) up to the
# ends of the 64-bit range, next to small ones, with and without a second addend
@pytest.mark.parametrize("log_n", [5, 10, 13, 14])
@pytest.mark.parametrize("bits", [[50, 45, 52], [61, 50, 54]])
def test_encryption_of_any_64_bit_integers(log_n, bits):
    import torch

    import paper_2601_15401_gb300 as G
    p = synth.make_params(log_n, bits, 1, 3)
    ctx, octx = G.Context.from_params(p), O.Ctx(p)
    N = p.N
    ends = [0, 1, -1, (1 << 61) - 1, 1 << 61, -(1 << 61), -(1 << 61) - 1, (1 << 62) + 5, -(1 << 62) - 7,
            (1 << 63) - 1, -(1 << 63), 12345678901234567]
    g = synth.rng(88, log_n)
    m = np.array([ends[i % len(ends)] for i in range(N)], dtype=np.int64)
    m[N // 2:] = g.integers(-(1 << 50), 1 << 50, size=N - N // 2)   # sets within the fast path too
    v, e0, e1 = synth.ternary_weight(g, N, N // 2), synth.gaussian(g, N), synth.gaussian(g, N)
    e0[3] = (1 << 62) + 3
    s, a, e = synth.ternary_secret(g, N), synth.uniform_residues(g, p.q, N), synth.gaussian(g, N)
    ws = torch.empty(ctx.encrypt_workspace_size() // 8, dtype=torch.uint64, device="cuda")
    pk = torch.empty((2, p.L, N), dtype=torch.uint64, device="cuda")
    ctx.public_key(torch.from_numpy(s).cuda(), dev(a), torch.from_numpy(e).cuda(), pk, ws)
    opk = O.public_key(octx, s, a, e)
    assert np.array_equal(host(pk), np.stack(opk))
    out = G.Tuple.wrap(torch.zeros((2, p.L, N), dtype=torch.uint64, device="cuda"))
    ctx.encrypt(*(torch.from_numpy(x).cuda() for x in (m, v, e0, e1)), pk, p.L, out, ws)
    ctx.check()
    assert np.array_equal(host(out.data), O.encrypt(octx, [int(x) for x in m], opk, v, e0, e1))
