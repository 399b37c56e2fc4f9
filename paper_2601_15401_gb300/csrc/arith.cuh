// Modular arithmetic by constants on 64-bit words, shared by the kernels and
// (compiled as plain C++) by the host tables and the host tests.
//
// A product x w mod q by a constant w takes a quotient estimate
// h ~ x w / q from a precomputed companion of w and returns
// r = x w - h q (mod 2^64), a small signed multiple-of-q remainder (Shoup's
// precomputed-quotient method with a signed, rounded quotient). What bounds
// every kernel built on it is the integer multiply pipe: a 32 x 32 -> 64-bit
// multiply-add holds it for four cycles per warp, a 32-bit one for two, and
// the compiler also places moves and two-operand adds on it. So the product
// is spelled in five wide and four narrow multiply-adds and nothing else on
// that pipe:
//   quotient   three wide (the fourth, low x low, would move h by less than
//              one; r absorbs it),
//   remainder  two wide and four narrow, all accumulating: x w + h (-q).
// Register-only streams on a GB300 (warp cycles per butterfly and scheduler):
// 35-36 for both butterflies below, against 49 / 51 for the exact-quotient
// forms with conditional subtractions (four-product high word, two separate
// low products).
//
// Lazy values are signed: r may be negative, sums and differences are plain
// 64-bit adds, and no correction is needed between butterflies while the
// bound below stays under 2^63. Two companions:
//   balanced   any q < 2^61, |x| < 2^63 - 2^33: |r| < q. w is taken in
//              about (-q/2, q/2), its quotient w/q as the signed 64-bit
//              fraction P = p1 2^32 + p0 with both halves signed, and x is
//              split with a signed low half.
//   halved     q < 2^53 (kSmallBits), |x| < 2^62: |r| < 2.25 q. w in
//              [0, q), P = w 2^63 / q, x split with an unsigned low half
//              (one operation less); the quotient counts multiples of 2q.
#pragma once
#include <cstdint>

#if defined(__CUDACC__)
#define CKKS_HD __host__ __device__ __forceinline__
#else
#define CKKS_HD inline
#endif

typedef unsigned long long u64;
typedef long long i64;
typedef uint32_t u32;

// Primes below 2^kSmallBits take the halved companion and the uncorrected
// butterflies ("small"); the others ("big") the balanced one. With 53 bits a
// radix-16 inverse pass over inputs below 18 q (sums and differences up to
// 288 q) stays below 2^62.
constexpr int kSmallBits = 53;
CKKS_HD bool small_prime(u64 q) { return (q >> kSmallBits) == 0; }

// Shoup constant: w and its quotient companion (balanced form unless said
// otherwise), high half p1, low half p0.
struct Shoup {
    u64 w, wp;
};

CKKS_HD u32 lo32(u64 x) { return (u32)x; }
CKKS_HD u32 hi32(u64 x) { return (u32)(x >> 32); }

CKKS_HD u64 pack64(u32 lo, u32 hi) {
#if defined(__CUDA_ARCH__)
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
#else
    return ((u64)hi << 32) | lo;
#endif
}

// a b + c: unsigned and signed 32 x 32 -> 64-bit, and 32-bit
CKKS_HD u64 mad_wide(u32 a, u32 b, u64 c) {
#if defined(__CUDA_ARCH__)
    u64 r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (u64)a * b + c;
#endif
}

CKKS_HD u64 mad_wide_s(u32 a, u32 b, u64 c) {
#if defined(__CUDA_ARCH__)
    u64 r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (u64)((i64)(int32_t)a * (int32_t)b) + c;
#endif
}

CKKS_HD u32 mad_lo(u32 a, u32 b, u32 c) {
#if defined(__CUDA_ARCH__)
    u32 r;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
#else
    return a * b + c;
#endif
}

// Quotient estimates. v = the two cross products plus half a unit (rounding)
// plus an offset that keeps it non-negative as an unsigned word; the offset
// leaves through the high product's addend.
CKKS_HD u64 quot_balanced(u64 x, u64 wp) {
    const u32 x0 = lo32(x), x1 = hi32(x) + (x0 >> 31);  // x = x1 2^32 + (signed) x0
    u64 v = mad_wide_s(x0, hi32(wp), 0x8000000080000000ull);
    v = mad_wide_s(x1, lo32(wp), v);
    return mad_wide_s(x1, hi32(wp), 0xffffffff80000000ull) + (u64)hi32(v);
}

CKKS_HD u64 quot_halved(u64 x, u64 wp) {
    u64 v = mad_wide(lo32(x), hi32(wp), 0x4000000080000000ull);
    v = mad_wide_s(hi32(x), lo32(wp), v);
    return mad_wide_s(hi32(x), hi32(wp), 0xffffffffc0000000ull) + (u64)hi32(v);
}

// add + x w - h M (mod 2^64), nm = -M. With Q1, M = mult q for a prime
// q = 1 (mod 2^32) and mult 1 or 2: the low half of h M is then mult h
// itself, so the quotient product is one narrow multiply.
template <bool Q1, int MULT>
CKKS_HD u64 remainder_mad(u64 x, u64 w, u64 h, u64 nm, u64 add) {
    u64 r = mad_wide(lo32(x), lo32(w), add);
    if constexpr (Q1) {
        u32 t = mad_lo(lo32(x), hi32(w), hi32(r));
        t = mad_lo(hi32(x), lo32(w), t);
        // h M = mult h + (h0 Mh) 2^32 with M = Mh 2^32 + mult; -M = ~Mh 2^32 + (2^32 - mult)
        t = mad_lo(lo32(h), hi32(nm) + 1u, t);
        r = pack64(lo32(r), t) - h;
        return MULT == 2 ? r - h : r;
    } else {
        r = mad_wide(lo32(h), lo32(nm), r);
        u32 t = mad_lo(lo32(x), hi32(w), hi32(r));
        t = mad_lo(hi32(x), lo32(w), t);
        t = mad_lo(lo32(h), hi32(nm), t);
        t = mad_lo(hi32(h), lo32(nm), t);
        return pack64(lo32(r), t);
    }
}

// x w mod q as a signed value in (-q, q); balanced companion, |x| < 2^63 - 2^33.
template <bool Q1>
CKKS_HD u64 shoup_signed(u64 x, u64 w, u64 wp, u64 q) {
    return remainder_mad<Q1, 1>(x, w, quot_balanced(x, wp), 0ull - q, 0ull);
}

// (-q, q) -> [0, q)
CKKS_HD u64 lift_sign(u64 r, u64 q) { return (i64)r < 0 ? r + q : r; }

// x w mod q in [0, q).
template <bool Q1>
CKKS_HD u64 shoup_t(u64 x, u64 w, u64 wp, u64 q) {
    return lift_sign(shoup_signed<Q1>(x, w, wp, q), q);
}
CKKS_HD u64 shoup(u64 x, u64 w, u64 wp, u64 q) { return shoup_t<false>(x, w, wp, q); }

// Cooley-Tukey butterfly (X, Y) <- (X + w Y, X - w Y) on signed lazy values:
// each stage adds less than 2.25 q (small) or q (big) to the bound. The
// second output is 2 X - X' (three-operand adds stay off the multiply pipe).
template <bool SMALL, bool Q1>
CKKS_HD void ct_bfly(u64 &X, u64 &Y, u64 w, u64 wp, u64 q) {
    const u64 x = X;
    if constexpr (SMALL) X = remainder_mad<Q1, 2>(Y, w, quot_halved(Y, wp), 0ull - 2 * q, x);
    else X = remainder_mad<Q1, 1>(Y, w, quot_balanced(Y, wp), 0ull - q, x);
    Y = x + x - X;
}

// Gentleman-Sande butterfly (X, Y) <- (X + Y, (X - Y) w): the sum doubles the
// bound, the product is below 2.25 q (small) or q (big).
template <bool SMALL, bool Q1>
CKKS_HD void gs_bfly(u64 &X, u64 &Y, u64 w, u64 wp, u64 q) {
    const u64 x = X, d = X - Y;
    X = x + x - d;
    if constexpr (SMALL) Y = remainder_mad<Q1, 2>(d, w, quot_halved(d, wp), 0ull - 2 * q, 0ull);
    else Y = remainder_mad<Q1, 1>(d, w, quot_balanced(d, wp), 0ull - q, 0ull);
}

// |x| <= 2 c -> |x| <= c, the same residue for c a multiple of q.
CKKS_HD u64 fold_sign(u64 x, u64 c) { return x + ((i64)x < 0 ? c : 0ull - c); }

// Reduction of small multiples of q: with b the bit length of q,
// shift = max(0, b - 11) and mul = floor(2^(b + 12) / q) (between 2^12 and
// 2^13), floor(u / q) for u < 256 q is ((u >> shift) mul) >> (b + 12 - shift)
// or one more: the truncations lose less than 2^-10 + 256 2^-12 of a unit.
struct Canon {
    u32 mul, shifts;  // shifts = shift | (b + 12 - shift) << 8
};

CKKS_HD Canon make_canon(u64 q) {
    int b = 0;
    while (b < 64 && (q >> b)) ++b;
    Canon c;
    const int s = b > 11 ? b - 11 : 0;
    // floor(2^(b + 12) / q) by long division (13 quotient bits; q < 2^61)
    u64 rem = (u64)1 << (b - 1), quo = 0;
    if (rem >= q) rem -= q, quo = 1;
    for (int i = 0; i < 13; ++i) {
        rem <<= 1;
        quo <<= 1;
        if (rem >= q) rem -= q, quo |= 1;
    }
    c.mul = (u32)quo;
    c.shifts = (u32)s | (u32)(b + 12 - s) << 8;
    return c;
}

// u - floor(u / q) q or one q more, u < 256 q (unsigned 64-bit): in [0, 2q).
CKKS_HD u64 reduce_near(u64 u, u64 q, Canon c) {
    const u32 k = ((u32)(u >> (c.shifts & 63)) * c.mul) >> (c.shifts >> 8);
    const u64 nq = 0ull - q;
    const u64 r = mad_wide(k, lo32(nq), u);
    return pack64(lo32(r), mad_lo(k, hi32(nq), hi32(r)));
}

// The same for u < 1024 q (wide product for the quotient): in [0, 2q).
CKKS_HD u64 reduce_far(u64 u, u64 q, Canon c) {
    const u32 k = (u32)(mad_wide((u32)(u >> (c.shifts & 63)), c.mul, 0ull) >> (c.shifts >> 8));
    const u64 nq = 0ull - q;
    const u64 r = mad_wide(k, lo32(nq), u);
    return pack64(lo32(r), mad_lo(k, hi32(nq), hi32(r)));
}

// A forward transform's signed lazy value (small: |v| < 128 q; big: |v| < 8 q
// below 2^60, < 4 q above) -> [0, q).
template <bool SMALL>
CKKS_HD u64 canonical(u64 v, u64 q, Canon c) {
    const u64 off = SMALL ? q << 7 : (q >> 60 ? q << 2 : q << 3);
    const u64 r = reduce_near(v + off, q, c);
    return r >= q ? r - q : r;
}

// ---------------------------------------------------------------------------
// dot products by limbs
// ---------------------------------------------------------------------------
// Operands v = v0 + v1 2^SB with both limbs below 2^30; a product is three
// wide multiply-adds, one per sum (Karatsuba's middle term), with no carry
// between them:
//   s0 = sum a0 b0,  s1 = sum a1 b1,  sx = sum (a0 + a1)(b0 + b1),
//   a . b = s0 + (sx - s0 - s1) 2^SB + s1 2^(2 SB),
// exact while s0, s1 and the middle sum a0 b1 + a1 b0 stay below 2^64 (sx may
// wrap: only the difference counts). SB = 30 (operands below 2^60): at most 8
// terms. SB = 27 (small primes: limbs below 2^27 and 2^26): at most 512
// terms. Measured as a register-only stream on a GB300: 15.8 warp cycles per
// product and scheduler, against 33-40 for a 64 x 64 -> 128-bit product (high
// and low words separately) added with carry.
constexpr int kLimbTerms30 = 8;
constexpr int kLimbTerms27 = 512;

struct Limbs {
    u32 lo, hi, sum;
};

template <int SB>
CKKS_HD Limbs split_limbs(u64 v) {
    Limbs l;
    l.lo = (u32)v & ((1u << SB) - 1);
    l.hi = (u32)(v >> SB);
    l.sum = l.lo + l.hi;
    return l;
}

// a word holding its own limbs (low limb in the low half)
template <int SB>
CKKS_HD u64 pack_limbs(u64 v) {
    return ((v >> SB) << 32) | (v & ((1u << SB) - 1));
}
CKKS_HD Limbs packed_limbs(u64 w) { return Limbs{lo32(w), hi32(w), lo32(w) + hi32(w)}; }

struct DotLimbs {
    u64 s0, s1, sx;
    CKKS_HD void zero() { s0 = s1 = sx = 0; }
    CKKS_HD void mac(const Limbs &a, const Limbs &b) {
        s0 = mad_wide(a.lo, b.lo, s0);
        s1 = mad_wide(a.hi, b.hi, s1);
        sx = mad_wide(a.sum, b.sum, sx);
    }
    // (the sum + a multiple of q) / 2^(2 SB): Montgomery reduction by limbs, two
    // steps of SB bits (R = 2^(2 SB)) that take one narrow and two wide
    // multiplies each and no 64 x 64-bit product. q0, q1: q's limbs;
    // nqi = -q^-1 mod 2^SB. In [0, sum / 2^(2 SB) + q + 1).
    template <int SB>
    CKKS_HD u64 redc(u32 q0, u32 q1, u32 nqi) const {
        constexpr u32 M = (1u << SB) - 1;
        const u64 x = sx - s0 - s1;
        const u32 m0 = mad_lo(lo32(s0), nqi, 0u) & M;
        const u64 a = mad_wide(m0, q0, s0) >> SB;
        const u64 b = mad_wide(m0, q1, (u64)(lo32(x) & M)) + a;
        const u32 m1 = mad_lo(lo32(b), nqi, 0u) & M;
        const u64 c = mad_wide(m1, q0, b) >> SB;
        return mad_wide(m1, q1, s1) + (x >> SB) + c;
    }
    // SB = 30: brings the sums of up to 7 terms (or of a folded value, worth
    // one, and 6 terms) back to a value below 2 q 2^60 + 2^60: the middle sum's
    // high part and the high sum, reduced mod q, and two low limbs.
    CKKS_HD void fold(u64 q, Canon c) {
        u64 x = sx - s0 - s1;
        x += s0 >> 30;
        s0 &= (1u << 30) - 1;
        // operands are below q, their high limbs at most q / 2^30, so the high
        // sum is at most 7 q^2 / 2^60 (after a fold 2 q + 6 q^2 / 2^60) and the
        // middle one's high part 14 q / 2^30 + 8: below 256 q for every q < 2^60
        s1 = reduce_near(s1 + (x >> 30), q, c);
        x &= (1u << 30) - 1;
        sx = x + s0 + s1;
    }
    // the sum as hi 2^64 + lo
    template <int SB>
    CKKS_HD void value(u64 &hi, u64 &lo) const {
        const u64 x = sx - s0 - s1;
        u64 l = s0 + (x << SB);
        u64 h = (x >> (64 - SB)) + (s1 >> (64 - 2 * SB)) + (l < s0 ? 1ull : 0ull);
        const u64 m = l + (s1 << (2 * SB));
        h += m < l ? 1ull : 0ull;
        lo = m;
        hi = h;
    }
};

// ---------------------------------------------------------------------------
// host: companions
// ---------------------------------------------------------------------------
// (w, balanced companion) for 0 <= w < q: w (mod 2^64, possibly negative) and
// P = round(w 2^64 / q) as p1 2^32 + p0 with p1, p0 signed 32-bit.
inline Shoup make_shoup(u64 w, u64 q) {
    typedef unsigned __int128 u128;
    const u128 num = ((u128)w << 64) + q / 2;
    u128 P = num / q;  // <= 2^64
    Shoup s;
    s.w = w;
    // the halves of the signed value nearest zero that p1 can hold: P in
    // [-2^63 - 2^31, 2^63 - 2^31)
    if (P >= ((u128)1 << 63) - ((u128)1 << 31)) {
        P -= (u128)1 << 64;
        s.w = w - q;
    }
    const u32 p0 = (u32)(u64)P;
    const u32 p1 = (u32)((u64)((__int128)(P - (u128)(__int128)(int32_t)p0) >> 32));
    s.wp = ((u64)p1 << 32) | p0;
    return s;
}

// (w, halved companion) for 0 <= w < q < 2^kSmallBits: P = round(w 2^63 / q).
inline Shoup make_shoup_halved(u64 w, u64 q) {
    typedef unsigned __int128 u128;
    u128 P = (((u128)w << 63) + q / 2) / q;
    Shoup s;
    s.w = w;
    if (P >= ((u128)1 << 63) - ((u128)1 << 31)) {  // p1 would be 2^31: take w - q
        P -= (u128)1 << 63;
        s.w = w - q;
    }
    const u32 p0 = (u32)(u64)P;
    const u32 p1 = (u32)((u64)((__int128)(P - (u128)(__int128)(int32_t)p0) >> 32));
    s.wp = ((u64)p1 << 32) | p0;
    return s;
}

// the companion of an NTT twiddle of prime q
inline Shoup make_twiddle(u64 w, u64 q) { return small_prime(q) ? make_shoup_halved(w, q) : make_shoup(w, q); }
