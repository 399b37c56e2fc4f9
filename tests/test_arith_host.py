"""The kernels' modular arithmetic (csrc/arith.cuh) compiled as plain C++ and
compared with 128-bit integers at the edges of its ranges: products by a
constant with both companions (operands up to the stated bounds, constants
next to 0, q/2 and q, primes of every size and of the form h 2^32 + 1), the
reductions of small multiples of q, and the dot products by limbs."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "paper_2601_15401_gb300/csrc/arith.cuh"
#include <cstdio>
#include <random>
typedef unsigned __int128 u128;
typedef __int128 i128;
static u64 smod(i128 x, u64 q) { i128 r = x % (i128)q; return (u64)(r < 0 ? r + q : r); }
static long bad = 0;
static void check(bool ok, const char *what, u64 q, u64 w, i64 x) {
    if (!ok && bad++ < 8) printf("%s q=%llu w=%llu x=%lld\n", what, q, w, x);
}
template <bool Q1> static void products(u64 q, u64 w, i64 x, int m) {
    const Shoup s = make_shoup(w, q);
    const i64 r = (i64)shoup_signed<Q1>((u64)x, s.w, s.wp, q);
    check((r < 0 ? 0ull - (u64)r : (u64)r) < q && smod(r, q) == smod((i128)smod(x, q) * w, q), "balanced", q, w, x);
    if (!small_prime(q)) return;
    const i64 lim = (1ll << 62) - 1, y = m == 0 ? lim : m == 1 ? -lim : x % lim;
    const Shoup h = make_shoup_halved(w, q);
    const i64 t = (i64)remainder_mad<Q1, 2>((u64)y, h.w, quot_halved((u64)y, h.wp), 0ull - 2 * q, 0);
    check((double)(t < 0 ? -t : t) < 2.25 * (double)q && smod(t, q) == smod((i128)smod(y, q) * w, q), "halved", q, w, y);
}
template <int SB> static void dots(u64 q, u64 qb, int terms, std::mt19937_64 &g) {
    DotLimbs d;
    d.zero();
    u128 sum = 0;
    for (int i = 0; i < terms; ++i) {
        const u64 a = g() % 3 ? q - 1 - g() % 5 % q : g() % q, b = g() % 3 ? qb - 1 - g() % 5 % qb : g() % qb;
        d.mac(split_limbs<SB>(a), packed_limbs(pack_limbs<SB>(b)));
        sum += (u128)a * b;
    }
    u64 hi, lo;
    d.value<SB>(hi, lo);
    check(hi == (u64)(sum >> 64) && lo == (u64)sum, "dot", q, qb, terms);
    // Montgomery reduction of the sum by limbs modulo the prime qb: r 2^(2 SB) = sum
    // (mod qb), r <= sum / 2^(2 SB) + qb
    u64 inv = qb;
    for (int i = 0; i < 6; ++i) inv *= 2 - qb * inv;
    const u64 r = d.redc<SB>((u32)qb & ((1u << SB) - 1), (u32)(qb >> SB), 0u - (u32)inv);
    const u128 R = ((u128)1 << (2 * SB)) % qb;
    check((u64)((u128)(r % qb) * (u64)R % qb) == (u64)(sum % qb) && (u128)r <= (sum >> (2 * SB)) + qb + 1, "redc", q, qb,
          terms);
}
int main() {
    std::mt19937_64 g(20);
    const u64 qs[] = {97, 12289, 65537, 1073479681ull, (1ull << 45) - 1, (1ull << 50) - 27 * 131072 + 1, (1ull << 52) + 1,
                      (1ull << 53) - 111, (1ull << 53) + 5, (1ull << 60) - 131071, (1ull << 60) + 131073,
                      (1ull << 61) - 1, (12345ull << 32) + 1, (200001ull << 32) + 1, ((1ull << 28) - 5 << 32) + 1,
                      ((1ull << 29) - 5 << 32) + 1};
    for (u64 q : qs) {
        const Canon c = make_canon(q);
        for (int it = 0; it < 60000; ++it) {
            u64 w = g() % q;
            if (it < 96) w = (it < 32 ? it : it < 64 ? q - 1 - (it - 32) % q : q / 2 + it - 80) % q;
            const i64 lim = 0x7fffffffffffffffll - (1ll << 33);
            const int m = it % 7;
            i64 x = (i64)g() % lim;
            if (m == 0) x = lim;
            if (m == 1) x = -lim;
            if (m == 2) x = (i64)(g() % q);
            if (m == 3) x = (x & ~0xffffffffll) | 0x80000000;
            if (m == 4) x >>= g() % 60;
            products<false>(q, w, x, m);
            if ((u32)q == 1) products<true>(q, w, x, m);
            if (small_prime(q)) {
                u64 u = m == 0 ? q * 256 - 1 : m == 1 ? q * (g() % 256) : m == 2 ? q * (g() % 255 + 1) - 1 : g() % (q * 256);
                u64 r = reduce_near(u, q, c);
                check(r < 2 * q && r % q == u % q, "near", q, u, 0);
                u = m == 0 ? q * 1024 - 1 : m == 1 ? q * (g() % 1024) : g() % (q * 1024);
                r = reduce_far(u, q, c);
                check(r < 2 * q && r % q == u % q, "far", q, u, 0);
            }
            const u64 span = small_prime(q) ? 128 : q >> 60 ? 4 : 8;  // |v| < span q
            const i128 v = (i128)((((u128)g() << 64) | g()) % ((u128)span * 2 * q - 1)) - ((i128)span * q - 1);
            const u64 r = small_prime(q) ? canonical<true>((u64)(i64)v, q, c) : canonical<false>((u64)(i64)v, q, c);
            check(r == smod(v, q), "canonical", q, w, (i64)v);
        }
        for (int it = 0; it < 2000 && q < (1ull << 60); ++it) {
            const u64 qb = it % 2 ? q : (1ull << 60) - 131071;
            dots<30>(q, qb, 1 + it % kLimbTerms30, g);
            if (small_prime(q)) dots<27>(q, q, 1 + it % kLimbTerms27, g);
            // fold: 7 terms, then 6 at a time
            DotLimbs d;
            d.zero();
            u128 sum = 0;
            for (int i = 0; i < 7 + 6 * (it % 5); ++i) {
                const u64 a = q - 1 - g() % 7 % q, b = it % 3 ? q - 1 : g() % q;
                d.mac(split_limbs<30>(a), split_limbs<30>(b));
                sum = (sum + (u128)a * b) % q;
                if (i >= 6 && (i - 6) % 6 == 0) d.fold(q, c);
            }
            u64 hi, lo;
            d.value<30>(hi, lo);
            check(hi < q && (u64)((((u128)hi << 64) | lo) % q) == (u64)sum, "fold", q, it, 0);
        }
    }
    printf("bad %ld\n", bad);
    return bad ? 1 : 0;
}
"""


def test_arithmetic_against_128_bit_integers(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "arith.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "arith"
    subprocess.run([cxx, "-O2", "-std=c++17", "-w", "-I", ROOT, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
