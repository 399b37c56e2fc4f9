"""Workloads of the library, each one call (or the pair of calls that belong
together) through its public entry points on seeded synthetic data.

  listed()            the fixed cases
  draw(rng)           one more case of the same ranges
  prepare(case, seed) inputs, keys and handles a program holds before the call
  run(state)          one pass; returns every output
  work(case)          bytes and operations a pass cannot do without
  exact(case, seed)   outputs computed in plain numpy, where they are not residues

Parameter families are the repository's own: small (N = 2^10, four 50-bit q,
one 60-bit p, dnum 1), mid (60-bit q_0 and eleven 45-bit q, four 60-bit p,
dnum 3) and large (24 x 50-bit q, 8 x 60-bit p, dnum 3); `q1` takes primes
that are 1 (mod 2^32) instead of 1 (mod 2^17).
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2601_15401_gb300 as G
import synth

SCALE = 2.0 ** 50


def listed():
    return [
        # one small product, where launches and latency are the cost
        {"name": "mul_n1024_k3_b1", "kind": "mul", "family": "small", "log_n": 10, "k": 3, "level": 4, "batch": 1,
         "dropped": False, "q1": False},
        # many independent triples of the three-input setting in one call
        {"name": "mul_n16384_k3_b64", "kind": "mul", "family": "mid", "log_n": 14, "k": 3, "level": 12, "batch": 64,
         "dropped": False, "q1": False},
        # one request served alone, at a level it has been rescaled to (its
        # ciphertexts still carry the stride of a fresh one)
        {"name": "mul_n32768_k7_b1", "kind": "mul", "family": "large", "log_n": 15, "k": 7, "level": 17, "batch": 1,
         "dropped": True, "q1": False},
        # the flagship batch of the k-input setting, at its largest k
        {"name": "mul_n65536_k12_b16", "kind": "mul", "family": "large", "log_n": 16, "k": 12, "level": 24,
         "batch": 16, "dropped": False, "q1": False},
        # a smaller, odd batch on primes that are 1 (mod 2^32)
        {"name": "mul_n65536_k5_b7_q1", "kind": "mul", "family": "large", "log_n": 16, "k": 5, "level": 21,
         "batch": 7, "dropped": False, "q1": True},
        # products of every k and level together, as an executor replays them
        {"name": "wave_n32768_40", "kind": "wave", "log_n": 15, "count": 40, "mix": 11},
        # the standard two-input product, mid-chain (a ragged last digit)
        {"name": "mul2_n65536_b8", "kind": "mul2", "log_n": 16, "level": 13, "batch": 8},
        # slot rotation of a batch of fresh ciphertexts
        {"name": "rotate_n65536_b16", "kind": "rotate", "log_n": 16, "level": 24, "batch": 16, "r": 1},
        # a five-term tuple rescaled by three primes at once
        {"name": "rescale_n32768_p5_mu3", "kind": "rescale", "log_n": 15, "polys": 5, "level": 15, "mu": 3},
        # both directions of the transform at a small ring degree
        {"name": "ntt_n8192_p6", "kind": "ntt", "log_n": 13, "polys": 6, "level": 11},
        # a client's upload: slots encoded and encrypted
        {"name": "encrypt_n16384_b12", "kind": "encrypt", "log_n": 14, "level": 24, "batch": 12},
        # a client's download: results decrypted and decoded
        {"name": "decrypt_n32768_b9", "kind": "decrypt", "log_n": 15, "level": 5, "batch": 9},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    top = max(work(c)["flops"] for c in listed())
    while True:
        c = _draw(rng)
        if work(c)["flops"] <= top and _state_bytes(c) <= 30e9:
            return c


def _draw(rng):
    kind = rng.choice(["mul", "mul", "mul", "mul", "wave", "wave", "mul2", "rotate", "rescale", "ntt", "encrypt",
                       "decrypt"])
    log_n = rng.choice([14, 15, 16])
    if kind == "mul":
        fam = rng.choice(["small", "mid", "large", "large", "large"])
        q1 = rng.random() < 0.25 and fam == "large"
        if fam == "small":
            return {"kind": kind, "family": fam, "log_n": rng.choice([10, 11, 12, 13]), "k": rng.choice([2, 3, 4]),
                    "level": 4, "batch": _log_int(rng, 1, 32), "dropped": False, "q1": False}
        k = rng.randint(2, 12) if fam == "large" else rng.randint(2, 6)
        return {"kind": kind, "family": fam, "log_n": log_n, "k": k, "level": rng.randint(max(k, 6), _levels(fam)),
                "batch": _log_int(rng, 1, 16 << (16 - log_n)), "dropped": rng.random() < 0.4, "q1": q1}
    if kind == "wave":
        return {"kind": kind, "log_n": log_n, "count": _log_int(rng, 3, 20 << (16 - log_n)),
                "mix": rng.randrange(1 << 20)}
    if kind == "mul2":
        return {"kind": kind, "log_n": log_n, "level": rng.randint(3, 24), "batch": _log_int(rng, 1, 24)}
    if kind == "rotate":
        return {"kind": kind, "log_n": log_n, "level": rng.randint(2, 24), "batch": _log_int(rng, 1, 24),
                "r": rng.choice([1, -3, 7, 64, 513])}
    if kind == "rescale":
        level = rng.randint(6, 24)
        return {"kind": kind, "log_n": log_n, "polys": rng.randint(2, 13), "level": level, "mu": rng.randint(1, 4)}
    if kind == "ntt":
        return {"kind": kind, "log_n": rng.randint(8, 16), "polys": _log_int(rng, 1, 32), "level": rng.randint(1, 24)}
    return {"kind": kind, "log_n": log_n, "level": rng.randint(2, 24), "batch": _log_int(rng, 1, 32)}


def _levels(fam):
    return {"small": 4, "mid": 12, "large": 24}[fam]


# --------------------------------------------------------------------------
# what a program sets up once: parameters and the context
# --------------------------------------------------------------------------
@functools.lru_cache(maxsize=24)
def _params(fam, log_n, q1):
    cong = synth.Q1_CONGRUENCE if q1 else synth.NTT_CONGRUENCE
    if fam == "small":
        return synth.params_small(log_n=log_n, congruence=cong)
    if fam == "mid":
        return synth.params_mid(log_n=log_n, congruence=cong)
    return synth.params_large(log_n=log_n, congruence=cong)


@functools.lru_cache(maxsize=24)
def _context(fam, log_n, q1):
    return G.Context.from_params(_params(fam, log_n, q1))


def _of(case):
    key = (case.get("family", "large"), case["log_n"], case.get("q1", False))
    return _params(*key), _context(*key)


def _u64(*shape):
    return torch.empty(shape, dtype=torch.uint64, device="cuda")


def _ws(nbytes):
    return _u64(nbytes // 8 + 32)


def _residues(primes, prefix, N, seed):
    return synth.uniform_residues_torch(primes, prefix, N, seed, "cuda")


def _key_set(p, ctx, t_max, seed):
    """Evaluation keys of t = 2..t_max: pairs of uniform residues, as keys are."""
    keys = _residues(list(p.q) + list(p.p), (t_max - 1, p.dnum, 2), p.N, seed * 7919 + 5)
    return ctx.evk_set(t_max, keys)


def _ciphertexts(p, count, level, dropped, seed):
    stride = p.L if dropped else level
    data = _residues(p.q[:stride], (count, 2), p.N, seed)
    return data, [G.Tuple(data[i], 2, level, stride) for i in range(count)]


def _gauss(g, shape):
    return np.clip(np.rint(g.normal(0.0, 3.2, size=shape)), -19, 19).astype(np.int64)


def _ternary(g, shape):
    return g.integers(-1, 2, size=shape, dtype=np.int64)


def _client_draw(case, seed):
    """Secret, public-key error, messages and encryption noise of a client."""
    g = np.random.default_rng([seed, case["log_n"], case["batch"], case["level"]])
    N, B = 1 << case["log_n"], case["batch"]
    d = {"s": _ternary(g, N), "e": _gauss(g, N), "v": _ternary(g, (B, N)), "e0": _gauss(g, (B, N)),
         "e1": _gauss(g, (B, N))}
    # slots uniform in the unit disk; their encoding has coefficients of this spread
    d["z"] = np.sqrt(g.random((B, N // 2))) * np.exp(2j * np.pi * g.random((B, N // 2)))
    d["m"] = np.rint(g.normal(0.0, SCALE * math.sqrt(0.5 / N), size=(B, N))).astype(np.int64)
    return d


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _mix(case):
    """(k, level) of every product of a wave: k uniform in 2..12, level in k..24."""
    import random
    r = random.Random(case["mix"])
    out = []
    for _ in range(case["count"]):
        k = r.randint(2, 12)
        out.append((k, r.randint(max(k, 5), 24)))
    return out


# --------------------------------------------------------------------------
# prepare / run
# --------------------------------------------------------------------------
def prepare(case, seed):
    p, ctx = _of(case)
    kind, N = case["kind"], p.N
    st = {"kind": kind, "ctx": ctx}
    if kind == "mul":
        k, B, level = case["k"], case["batch"], case["level"]
        st["evk"] = _key_set(p, ctx, k, seed)
        st["data"], cts = _ciphertexts(p, B * k, level, case["dropped"], seed)
        st["cts"] = [cts[b * k:(b + 1) * k] for b in range(B)]
        ol = level - ctx.plan_describe(k)["depth"]
        st["out"] = _u64(B, 2, ol, N)
        st["outs"] = [G.Tuple(st["out"][b], 2, ol, ol) for b in range(B)]
        st["ws"] = _ws(ctx.workspace_size(k, level, B))
    elif kind == "wave":
        mix = _mix(case)
        st["evk"] = _key_set(p, ctx, 12, seed)
        items, st["data"], st["out"] = [], [], []
        for i, (k, level) in enumerate(mix):
            data, cts = _ciphertexts(p, k, level, False, seed * 1009 + i)
            ol = level - ctx.plan_describe(k)["depth"]
            out = _u64(2, ol, N)
            st["data"].append(data)
            st["out"].append(out)
            items.append((cts, G.Tuple(out, 2, ol, ol), None))
        st["wave"] = G.Wave(ctx, items, st["evk"])
        st["tables"], st["scratch"] = st["wave"].buffers()
    elif kind == "mul2":
        B, level = case["batch"], case["level"]
        st["evk"] = _key_set(p, ctx, 2, seed)
        st["da"], st["a"] = _ciphertexts(p, B, level, False, seed)
        st["db"], st["b"] = _ciphertexts(p, B, level, False, seed + 104729)
        st["out"] = _u64(B, 2, level - 1, N)
        st["outs"] = [G.Tuple(st["out"][b], 2, level - 1, level - 1) for b in range(B)]
        st["ws"] = _ws(ctx.mul2_workspace_size(level, B))
    elif kind == "rotate":
        B, level = case["batch"], case["level"]
        st["g"] = ctx.galois_element(case["r"])
        st["evk"] = _key_set(p, ctx, 2, seed)
        st["data"], st["cts"] = _ciphertexts(p, B, level, False, seed)
        st["out"] = _u64(B, 2, level, N)
        st["outs"] = [G.Tuple(st["out"][b], 2, level, level) for b in range(B)]
        st["ws"] = _ws(ctx.rotate_workspace_size(level, B))
    elif kind == "rescale":
        np_, level, mu = case["polys"], case["level"], case["mu"]
        data = _residues(p.q[:level], (np_,), N, seed)
        st["t"] = G.Tuple(data, np_, level, level)
        st["mu"] = mu
        st["out"] = _u64(np_, level - mu, N)
        st["o"] = G.Tuple(st["out"], np_, level - mu, level - mu)
        st["ws"] = _ws(ctx.rescale_workspace_size(np_, level, mu))
    elif kind == "ntt":
        np_, level = case["polys"], case["level"]
        st["x"] = G.Tuple(_residues(p.q[:level], (np_,), N, seed), np_, level, level, 0)
        st["y"] = G.Tuple(_residues(p.q[:level], (np_,), N, seed + 1), np_, level, level, 1)
        st["fx"], st["fy"] = _u64(np_, level, N), _u64(np_, level, N)
    elif kind == "encrypt":
        B, level = case["batch"], case["level"]
        d = _client_draw(case, seed)
        for n in ("z", "v", "e0", "e1"):
            st[n] = _dev(d[n])
        st["pk"] = _public_key(p, ctx, d, seed)
        st["m"] = torch.empty((B, N), dtype=torch.int64, device="cuda")
        st["out"] = _u64(B, 2, level, N)
        st["outs"] = [G.Tuple(st["out"][b], 2, level, level) for b in range(B)]
        st["level"] = level
        st["ews"] = _ws(ctx.embed_workspace_size(B))
        st["ws"] = _ws(ctx.encrypt_batch_workspace_size(level, B))
    else:
        B, level = case["batch"], case["level"]
        d = _client_draw(case, seed)
        st["s"] = _dev(d["s"])
        pk = _public_key(p, ctx, d, seed)
        st["data"] = _u64(B, 2, level, N)
        st["cts"] = [G.Tuple(st["data"][b], 2, level, level) for b in range(B)]
        ws = _ws(ctx.encrypt_batch_workspace_size(level, B))
        ctx.encrypt_batch(_dev(d["m"]), _dev(d["v"]), _dev(d["e0"]), _dev(d["e1"]), pk, level, st["cts"], ws)
        st["m"] = torch.empty((B, N), dtype=torch.float64, device="cuda")
        st["z"] = torch.empty((B, N // 2), dtype=torch.complex128, device="cuda")
        st["ews"] = _ws(ctx.embed_workspace_size(B))
        st["ws"] = _ws(ctx.decrypt_batch_workspace_size(B))
        torch.cuda.synchronize()
    return st


def _public_key(p, ctx, d, seed):
    a = _residues(p.q, (), p.N, seed * 31 + 7)
    pk = _u64(2, p.L, p.N)
    ctx.public_key(_dev(d["s"]), a, _dev(d["e"]), pk, _ws(ctx.encrypt_workspace_size()))
    torch.cuda.synchronize()
    return pk


def run(st):
    ctx, kind = st["ctx"], st["kind"]
    if kind == "mul":
        ctx.mul_k_batch(st["cts"], st["evk"], st["outs"], st["ws"])
        return st["out"].view(torch.int64)
    if kind == "wave":
        st["wave"].run(st["tables"], st["scratch"])
        return [o.view(torch.int64) for o in st["out"]]
    if kind == "mul2":
        ctx.mul2_batch(st["a"], st["b"], st["evk"], st["outs"], st["ws"])
        return st["out"].view(torch.int64)
    if kind == "rotate":
        ctx.rotate_batch(st["cts"], st["g"], st["evk"], st["outs"], st["ws"])
        return st["out"].view(torch.int64)
    if kind == "rescale":
        ctx.rescale_multi(st["t"], st["mu"], st["o"], st["ws"])
        return st["out"].view(torch.int64)
    if kind == "ntt":
        x, y = st["x"], st["y"]
        ctx.ntt(x, G.Tuple(st["fx"], x.n_polys, x.level, x.level, 0))
        ctx.intt(y, G.Tuple(st["fy"], y.n_polys, y.level, y.level, 1))
        return [st["fx"].view(torch.int64), st["fy"].view(torch.int64)]
    if kind == "encrypt":
        ctx.encode(st["z"], SCALE, st["m"], st["ews"])
        ctx.encrypt_batch(st["m"], st["v"], st["e0"], st["e1"], st["pk"], st["level"], st["outs"], st["ws"])
        return [st["m"], st["out"].view(torch.int64)]
    ctx.decrypt_batch(st["cts"], st["s"], st["m"], st["ws"])
    ctx.decode(st["m"], SCALE, st["z"], st["ews"])
    return [st["m"], st["z"]]


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def _switch(p, n_keys, level):
    """Limb transforms and other modular products per coefficient of one key
    switch of n_keys polynomials at `level` (no rescale)."""
    digits = [min(level, (b + 1) * p.alpha) - b * p.alpha for b in range(-(-level // p.alpha))]
    transforms = n_keys * (level + sum(level - d + p.K for d in digits)) + 2 * (p.K + level)
    products = n_keys * sum(d * (level - d + p.K) for d in digits)      # ModUp
    products += 2 * n_keys * len(digits) * (level + p.K)                # key products
    products += 2 * p.K * level                                         # ModDown
    return transforms, products


def _product(p, k, level):
    """(operations, evaluation-key bytes) of one k-input product with the
    fewest limb transforms; two operations per modular product."""
    _, transforms = G.plan_optimize(k, "transforms", level, p.K, p.alpha)
    _, products = _switch(p, k - 1, level)
    depth = (k - 1).bit_length()
    digits = -(-(level - depth + 1) // p.alpha)
    return (2.0 * p.N * (transforms * p.log_n / 2 + products),
            8.0 * p.N * (k - 1) * digits * 2 * (level - depth + 1 + p.K))


def work(case):
    kind, log_n = case["kind"], case["log_n"]
    p = _params(case.get("family", "large"), log_n, case.get("q1", False))
    N, limb = p.N, 8.0 * p.N
    if kind in ("mul", "wave"):
        shapes = [(case["k"], case["level"])] * case["batch"] if kind == "mul" else _mix(case)
        flops = io = keys = 0.0
        seen = {}
        for k, level in shapes:
            if (k, level) not in seen:
                seen[k, level] = _product(p, k, level)
            f, kb = seen[k, level]
            flops += f
            io += limb * 2 * (k * level + level - (k - 1).bit_length())
            keys = max(keys, kb)
        return {"bytes": io + keys, "flops": flops}
    if kind in ("mul2", "rotate"):
        level, B = case["level"], case["batch"]
        transforms, products = _switch(p, 1, level)
        if kind == "mul2":
            transforms += 2 * level       # the rescale
            products += 4 * level
        polys = (4 * level + 2 * (level - 1)) if kind == "mul2" else 4 * level
        keys = limb * 2 * -(-level // p.alpha) * (level + p.K)
        return {"bytes": B * limb * polys + keys, "flops": 2.0 * B * N * (transforms * log_n / 2 + products)}
    if kind == "rescale":
        np_, level, mu = case["polys"], case["level"], case["mu"]
        return {"bytes": limb * np_ * (2 * level - mu),
                "flops": 2.0 * np_ * N * (level * log_n / 2 + (mu + 1) * (level - mu))}
    if kind == "ntt":
        limbs = case["polys"] * case["level"]
        return {"bytes": 4 * limb * limbs, "flops": 2.0 * 2 * limbs * N * log_n / 2}
    B, level = case["batch"], case["level"]
    fft = 2.5 * N * log_n * B * 2
    if kind == "encrypt":
        return {"bytes": limb * (B * (5 + 2 * level) + 2 * level), "flops": fft + 2.0 * B * N * level * (4 * log_n / 2 + 2)}
    return {"bytes": limb * (B * (4 + 2) + 1), "flops": fft + 2.0 * B * N * 2 * (log_n / 2 + 1)}


def _state_bytes(case):
    """Rough device bytes of a prepared state (drawn cases stay small)."""
    p = _params(case.get("family", "large"), case["log_n"], case.get("q1", False))
    limb = 8.0 * p.N
    if case["kind"] in ("mul", "wave"):
        shapes = [(case["k"], case["level"])] * case["batch"] if case["kind"] == "mul" else _mix(case)
        return sum(limb * (8 * k * level + (k - 1) * p.dnum * (level + p.K)) for k, level in shapes)
    return limb * 12 * case.get("batch", 1) * case["level"] * p.dnum


def exact(case, seed):
    if case["kind"] != "decrypt":
        return None
    d = _client_draw(case, seed)
    N = 1 << case["log_n"]
    ang = np.pi * np.arange(N) / N
    w = np.cos(ang) + 1j * np.sin(ang)

    def mul(a, b):
        """a b mod X^N + 1 of small integer polynomials (rounded, exact)."""
        return np.rint((np.fft.ifft(np.fft.fft(a * w) * np.fft.fft(b * w)) * np.conj(w)).real)

    # c_0 + c_1 s = m + v e + e_0 + e_1 s
    m = np.stack([d["m"][b] + mul(d["v"][b], d["e"]) + d["e0"][b] + mul(d["e1"][b], d["s"])
                  for b in range(case["batch"])]).astype(np.float64)
    Z = np.fft.ifft(m * w, axis=-1) * N
    pos = np.empty(N // 2, dtype=np.int64)
    x = 1
    for j in range(N // 2):
        pos[j] = (x - 1) // 2
        x = x * 5 % (2 * N)
    return [torch.from_numpy(m), torch.from_numpy(Z[:, pos] / SCALE)]
