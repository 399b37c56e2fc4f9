// Negacyclic NTT / INTT phase kernels over 64-bit NTT-friendly primes
// (device code; instantiated by ntt_[ut][fi][1].cu and ntt_whole_[ut][fi].cu, the
// host logic is in ntt.cu and phase_shape.h).
//
// The transform is the evaluation map A[i] = sum_j a_j psi^((2 brv(i)+1) j)
// (bit-reversed order), computed with Cooley-Tukey butterflies forward and
// Gentleman-Sande butterflies inverse (Section II; Eq. 7 and Algorithm 1
// use it between the coefficient and the NTT domain).
//
// GPU structure. N = N1 * N2 points split into a 2-D array with element
// e = c + k N2. The forward transform's first log2 N1 stages only pair
// elements of the same column c; its last log2 N2 stages only pair elements
// of the same row block [b N2, (b+1) N2). So the transform runs as two
// launches (column phase, block phase), each thread group loading whole
// columns or whole blocks, running their stages in registers and shared
// memory and writing back. The inverse runs the block phase first. N <= 2^12
// runs all stages in one launch, the whole limb in one CTA.
//
// Inside a phase the sub-transform of n = 2^LOGN points is done in passes of
// up to 4 stages: a thread holds 2^r points of one sub-problem in registers
// (radix-2^r), runs r butterfly stages on them and writes them back; passes
// are separated by a barrier. Butterflies are lazy on signed values
// (arith.cuh), with the corrections the prime's size asks for; a CTA works on
// one limb, so the choice is one uniform branch per CTA:
//   small primes (q < 2^53): forward values grow by 2.25 q a stage, at most
//     101 q over 16 stages (64 q of that from an Eq. 17 load), no correction
//     at all; inverse sums double every stage, so the one output of a pass
//     that is a sum at all its stages is brought to [0, 2q) after the pass
//     (the others end below 18 q, the next pass's sums below 288 q);
//   big primes: forward values grow by q a stage, and the intermediate between
//     the two phases is stored canonical (at most 8 stages, below 8 q; from
//     2^60 on the sums are folded every second stage); inverse sums are
//     folded to |x| <= q at every stage.
//
// Twiddles: psi^brv(k) with its companion for the forward, psi^-brv(k) for the
// inverse. The stage with m groups uses k = m + i for group i; in the block
// phase the global group index is b m_loc + i_loc and m = N1 m_loc, so
// k = m_loc (N1 + b) + i_loc. The table holds them in the order the passes read
// them (below).
//
// Element-wise work is fused into the global <-> shared copies: the load side
// can add two limbs or form the rescale combination of Eq. 17; the store side
// can scale (N^-1 and BConv / ModDown constants), finish ModDown (Eq. 5 with
// Eq. 11/12) or finish Algorithm 1 (A' = g A - B).
//
// Template parameters LM / SM fix the load / store mode at compile time
// (-1: read from the launch's spec at run time, N <= 2^8 only). A fixed mode
// keeps only the pointers and constants that mode uses alive, which is what
// lets the column kernels fit three or four CTAs per SM. A CTA finds its limb in
// the launch's uniform batch x polynomial x limb description (LimbJobs) or in a
// device table of NttJob entries (limbs of different products, levels and tree
// nodes in one launch).
//
// Bound by the integer multiply pipe: 74-81 % busy in the four phases of 384
// limbs at N = 2^16 (116 / 129 us forward columns / blocks, 122 / 140 inverse
// blocks / columns; 163 / 172 / 166 / 188 with the exact-quotient butterflies and
// run-time tiles before).
#pragma once
#include "common.cuh"
#include "internal.h"
#include "phase_shape.h"

namespace ckks {

// ---------------------------------------------------------------------------
// pass plan: LOGN stages in ceil(LOGN/4) passes of near-equal length
// ---------------------------------------------------------------------------
#ifndef CKKS_NTT_RMAX
#define CKKS_NTT_RMAX 4
#endif
template <int LOGN, int P>
struct Pass {
    static constexpr int NP = (LOGN + CKKS_NTT_RMAX - 1) / CKKS_NTT_RMAX;
    static constexpr int base = LOGN / NP;
    static constexpr int extra = LOGN % NP;
    static constexpr int len = base + (P < extra ? 1 : 0);
    static constexpr int start = P * base + (P < extra ? P : extra);
};

// Position of the twiddle of stage e of a pass (E0, R), its sub-problem group
// g and j < 2^e, within the pass's region of the twiddle table: the 2^R - 1
// twiddles a point set needs are 2^E0 entries apart, so one base pointer and
// constant offsets address them, and the threads of neighbouring groups read
// neighbouring entries (in stage order the same reads were 2^e entries
// apart: 16 to 32 cache lines per warp load, the L1 data stage 59 % busy in
// the forward block phase).
//   columns: region [2^E0, 2^(E0 + R)), entry (2^e - 1 + j) 2^E0 + g
//   block b: region [N1 2^E0, N1 2^(E0 + R)), entry (b (2^R - 1) + 2^e - 1 + j) 2^E0 + g
// (twiddle_slot in ntt.cu fills the table.)

// ---------------------------------------------------------------------------
// fused element-wise load / store with per-CTA base pointers
// ---------------------------------------------------------------------------
struct LoadCtx {
    int mode;
    const u64 *a, *b;      // limb base pointers (b: T limbs / z limbs / second addend)
    const Shoup *g;        // LD_EQ17: g[0..mu-1], g[mu] = self
    int mu, with_self, K, N;
    const u64 *cK;         // LD_BCONVK
    ModQ m;
};

struct StoreCtx {
    int mode;
    u64 *dst;
    const u64 *aux, *aux2;
    Shoup c;
    int K, N;
    const u64 *cK;
    ModQ m;
};

// uniform launches: limb (b, p, l) of the launch's views
__device__ __forceinline__ LoadCtx make_load(const LoadSpec &L, const LimbJobs &J, int N, int b, int p, int l,
                                             int prime, ModQ m) {
    LoadCtx c;
    c.mode = L.mode;
    c.N = N;
    c.m = m;
    c.mu = L.mu;
    c.with_self = L.with_self;
    c.K = L.K;
    const int slot = J.slot[l];
    c.a = L.a.ptr ? limb_ptr(L.a, b, p, slot, N) : nullptr;
    c.b = nullptr;
    c.g = nullptr;
    c.cK = nullptr;
    if (L.mode == LD_ADD) c.b = limb_ptr(L.b, b, p, slot, N);
    if (L.mode == LD_EQ17 || L.mode == LD_BCONVK) c.b = L.b.ptr + (i64)b * L.b.bstride + (i64)p * L.b.pstride;
    if (L.mode == LD_EQ17) c.g = L.g + (i64)l * (L.mu + 1);
    if (L.mode == LD_BCONVK) c.cK = L.cK + (i64)prime * CKKS_MAX_PRIMES;
    if (L.mode == LD_SIGNED) {
        c.a = L.sa[p] + (i64)b * N;
        c.b = L.sb[p] ? L.sb[p] + (i64)b * N : nullptr;
        c.g = L.one + prime;
    }
    return c;
}

__device__ __forceinline__ StoreCtx make_store(const StoreSpec &S, const LimbJobs &J, int N, int b, int p, int l,
                                               int prime, ModQ m) {
    StoreCtx c;
    c.mode = S.mode;
    c.N = N;
    c.m = m;
    c.K = S.K;
    const int ds = J.dslot[l];
    c.dst = limb_ptr(S.dst, b, p, ds, N);
    c.aux = nullptr;
    c.aux2 = nullptr;
    c.cK = nullptr;
    c.c = Shoup{0, 0};
    if (S.mode == ST_SCALE || S.mode == ST_MODDOWN || S.mode == ST_MRS) c.c = S.c[l * S.c_stride];
    if (S.mode == ST_MODDOWN) {
        c.aux = S.aux.ptr + (i64)b * S.aux.bstride + (i64)p * S.aux.pstride;
        c.cK = S.cK + (i64)prime * CKKS_MAX_PRIMES;
    }
    if (S.mode == ST_MRS || S.mode == ST_ADDSUB) c.aux = limb_ptr(S.aux, b, p, ds, N);
    if (S.mode == ST_ADDSUB) c.aux2 = limb_ptr(S.aux2, b, p, ds, N);
    return c;
}

// table launches: the limb's pointers come from its NttJob entry
__device__ __forceinline__ LoadCtx make_load(const LoadSpec &L, const NttJob &j, int N, ModQ m) {
    LoadCtx c;
    c.mode = L.mode;
    c.N = N;
    c.m = m;
    c.mu = j.mu;
    c.with_self = j.with_self;
    c.K = L.K;
    c.a = j.a;
    c.b = j.b;
    c.g = j.g;
    c.cK = L.mode == LD_BCONVK ? L.cK + (i64)j.prime * CKKS_MAX_PRIMES : nullptr;
    return c;
}

__device__ __forceinline__ StoreCtx make_store(const StoreSpec &S, const NttJob &j, int N, ModQ m) {
    StoreCtx c;
    c.mode = S.mode;
    c.N = N;
    c.m = m;
    c.K = S.K;
    c.dst = j.dst;
    c.aux = j.aux;
    c.aux2 = j.aux2;
    c.c = (S.mode == ST_SCALE || S.mode == ST_MODDOWN || S.mode == ST_MRS) ? *j.c : Shoup{0, 0};
    c.cK = S.mode == ST_MODDOWN ? S.cK + (i64)j.prime * CKKS_MAX_PRIMES : nullptr;
    return c;
}

// a + b of an Eq. 17 sum: lazy signed for small primes (at most 64 terms
// below q each), canonical for the others
template <bool SMALL>
__device__ __forceinline__ u64 eq17_add(u64 s, u64 r, u64 q) {
    return SMALL ? s + r : add_mod(s, lift_sign(r, q), q);
}
template <bool SMALL>
__device__ __forceinline__ u64 eq17_sub(u64 r, u64 s, u64 q) {
    return SMALL ? r - s : sub_mod(lift_sign(r, q), s, q);
}

// any signed 64-bit integer mod q (canonical); `one`: the constant 1
template <bool Q1>
__device__ __forceinline__ u64 signed_mod(u64 v, Shoup one, u64 q) {
    // v = 4 (v >> 2) + (v & 3): v itself may be beyond the product's range
    u64 r = shoup_t<Q1>((u64)((i64)v >> 2), one.w, one.wp, q);
    r = add_mod(r, r, q);
    r = add_mod(r, r, q);
    return add_mod(r, shoup_t<Q1>(v & 3, one.w, one.wp, q), q);
}

// out[u] = sum_i z_i[u DIST] c_i R^-1 mod q over the K limbs z_i (N apart) of the
// P basis, for G elements whose loads are in flight together. The sum of the
// P primes is below 2^64 (context check), so the high word stays below q.
template <int G, int DIST, bool Q1>
__device__ __forceinline__ void scaled_bconv(u64 (&out)[G], const u64 *z, int N, const u64 *cK, int K, ModQ m) {
    Acc128Lazy acc[G];
#pragma unroll
    for (int u = 0; u < G; ++u) acc[u].zero();
    for (int i = 0; i < K; ++i) {
        const u64 c = cK[i];
        u64 v[G];
#pragma unroll
        for (int u = 0; u < G; ++u) v[u] = z[(i64)i * N + u * DIST];
#pragma unroll
        for (int u = 0; u < G; ++u) acc[u].mac(v[u], c);
    }
#pragma unroll
    for (int u = 0; u < G; ++u) out[u] = redc_t<Q1>(acc[u].hi, acc[u].lo, m);
}

template <int LM, bool SMALL, bool Q1>
__device__ __forceinline__ u64 load_elem(const LoadCtx &c, int e) {
    const u64 q = c.m.q;
    const int mode = LM >= 0 ? LM : c.mode;
    switch (mode) {
    case LD_ADD:
        return add_mod(c.a[e], c.b[e], q);
    case LD_EQ17: {
        // sum_t g_t T_t (mod q); with the self term: g_self a - sum
        u64 s = 0;
        for (int t = 0; t < c.mu; ++t)
            s = eq17_add<SMALL>(s, shoup_signed<Q1>(c.b[(i64)t * c.N + e], c.g[t].w, c.g[t].wp, q), q);
        if (c.with_self) s = eq17_sub<SMALL>(shoup_signed<Q1>(c.a[e], c.g[c.mu].w, c.g[c.mu].wp, q), s, q);
        return s;
    }
    case LD_BCONVK: {
        u64 r[1];
        scaled_bconv<1, 1, Q1>(r, c.b + e, c.N, c.cK, c.K, c.m);
        return r[0];
    }
    case LD_SIGNED: {
        const Shoup one = *c.g;
        const u64 v = signed_mod<Q1>(c.a[e], one, q);
        return c.b ? add_mod(v, signed_mod<Q1>(c.b[e], one, q), q) : v;
    }
    default:
        return c.a[e];
    }
}

template <int SM, bool SMALL, bool Q1>
__device__ __forceinline__ void store_elem(const StoreCtx &c, int e, u64 v, bool fwd) {
    const u64 q = c.m.q;
    const int mode = SM >= 0 ? SM : c.mode;
    switch (mode) {
    case ST_LAZY:
        c.dst[e] = !SMALL && fwd ? canonical<SMALL>(v, q, c.m.canon) : v;
        break;
    case ST_SCALE:
        c.dst[e] = shoup_t<Q1>(v, c.c.w, c.c.wp, q);
        break;
    case ST_MODDOWN: {
        // c* = v N^-1 - sum_i z_i [p_i^-1 R]_q  (Eq. 5 with Eq. 11 / 12)
        u64 r[1];
        scaled_bconv<1, 1, Q1>(r, c.aux + e, c.N, c.cK, c.K, c.m);
        c.dst[e] = sub_mod(shoup_t<Q1>(v, c.c.w, c.c.wp, q), r[0], q);
        break;
    }
    case ST_MRS:
        // Algorithm 1, last step: A' = g^{mu,L-1} A - B
        c.dst[e] = sub_mod(shoup_t<Q1>(c.aux[e], c.c.w, c.c.wp, q), canonical<SMALL>(v, q, c.m.canon), q);
        break;
    case ST_ADDSUB:
        c.dst[e] = sub_mod(add_mod(c.aux[e], c.aux2[e], q), canonical<SMALL>(v, q, c.m.canon), q);
        break;
    default:  // ST_REDUCE
        c.dst[e] = canonical<SMALL>(v, q, c.m.canon);
        break;
    }
}

// ---------------------------------------------------------------------------
// one pass of a phase
// ---------------------------------------------------------------------------
// Threads. Every thread takes 16 points of a sub-problem (n >= 16):
//   columns: groups of 16 columns x n / 16 point sets, 16 adjacent columns
//            fastest, so every access to global memory is whole 128-byte row
//            segments; the tile is [n][16] per group; passes are separated by
//            __syncthreads;
//   blocks:  n / 16 threads per block, all in one warp, so passes are
//            separated by __syncwarp and warps never wait for each other; the
//            tile is [n + n / 16] per block (one pad word per 16).
// The geometry is fixed at compile time: every address within a thread's
// point set is one base plus constant offsets.
//   whole:   N <= 2^12 takes one launch for all stages: one CTA of n / 16
//            threads holds a limb (N >= 2^9), or a warp does (a block phase
//            with N1 = 1, kTinyLimbs warps per CTA).

// elements whose sums over the K z-limbs run together
#ifndef CKKS_NTT_MODDOWN_GROUP
#define CKKS_NTT_MODDOWN_GROUP 4
#endif

template <int LOGN, int LOGN2, int SH>
struct Geo {
    static constexpr int n = 1 << LOGN;
    static constexpr int sets = n >= 16 ? n / 16 : 1;               // threads per sub-problem
    static constexpr int group = SH == COLS ? 16 * sets : sets;     // threads per tile unit (16 columns / one block)
    static constexpr int unit = SH == COLS ? 16 * n : n + n / 16;   // shared words per tile unit
    static constexpr int stride = SH == COLS ? 1 << LOGN2 : 1;      // elements between neighbouring points in memory
    // blocks per warp (one where the block is the whole limb, N <= 2^8)
    static constexpr int warp_blocks = SH == BLOCKS && LOGN2 != 0 ? 32 / sets : 1;
    // bytes of a warp's part of a block-phase CTA: its blocks, then their n - 1 twiddles each
    static constexpr int warp_data = (warp_blocks * unit + 1) & ~1;  // words (even: the twiddles take 16-byte copies)
    static constexpr int warp_bytes = warp_data * 8 + warp_blocks * (n - 1) * 16;
    // shared offset of point pt relative to the thread's sub-problem; additive
    // over disjoint bit ranges of pt
    static __device__ __forceinline__ constexpr int off(int pt) { return SH == COLS ? pt * 16 : pt + (pt >> 4); }
};

// Asynchronous 16-byte copy into shared memory (no registers held while the
// load is in flight); groups complete in the order they were committed.
__device__ __forceinline__ void async_copy16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((u32)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}

template <int SH>
__device__ __forceinline__ void pass_sync() {
    if (SH == BLOCKS) __syncwarp();
    else __syncthreads();
}

// Whether a pass reads / writes global memory itself: always for columns, for
// blocks where it touches at least 8 consecutive words per sub-problem (the
// other side is staged through shared memory by the warp).
template <int LOGN, int SH, int P>
struct PassAccess {
    static constexpr int t_min = (1 << LOGN) >> (Pass<LOGN, P>::start + Pass<LOGN, P>::len);
    static constexpr bool direct = SH == COLS || t_min >= 8;
};

// R stages of butterflies on the 2^R points of one set; tw: the set's first
// twiddle, entries 2^E0 apart.
template <int R, int E0, bool FWD, bool SMALL, bool Q1, bool LONG>
__device__ __forceinline__ void set_stages(u64 (&x)[1 << R], const ulonglong2 *tw, u64 q) {
    constexpr int EL = 1 << R;
    if (FWD && !SMALL && LONG && E0 > 0 && !(q >> 60)) {
        // more than 8 stages in one phase: |x| < 8 q at every pass's end, so
        // folded to 4 q here the next pass ends below 8 q again
#pragma unroll
        for (int k = 0; k < EL; ++k) x[k] = fold_sign(x[k], q << 2);
    }
#pragma unroll
    for (int st = 0; st < R; ++st) {
        const int ep = FWD ? st : R - 1 - st;
        const int h = EL >> (ep + 1);
        if (FWD && !SMALL && ep % 2 == 0 && (q >> 60)) {
            // |x| < 4 q: two more stages after the fold stay below 4 q < 2^63
#pragma unroll
            for (int k = 0; k < EL; ++k)
                if ((k & h) == 0) x[k] = fold_sign(x[k], q << 1);
        }
#pragma unroll
        for (int k = 0; k < EL; ++k) {
            if ((k & h) == 0) {
                const ulonglong2 w = tw[((1 << ep) - 1 + (k >> (R - ep))) << E0];
                if (FWD) {
                    ct_bfly<SMALL, Q1>(x[k], x[k + h], w.x, w.y, q);
                } else {
                    gs_bfly<SMALL, Q1>(x[k], x[k + h], w.x, w.y, q);
                    if (!SMALL) x[k] = fold_sign(x[k], q);
                }
            }
        }
    }
}

// Loads of one point set from global memory: elements e + k dist, fused. The
// loads of all points are in flight together (for Eq. 17 term by term: a
// loop over the terms inside each element's load had one load in flight).
template <int EL, int DIST, int LM, bool SMALL, bool Q1>
__device__ __forceinline__ void load_set(u64 (&x)[EL], const LoadCtx &lc, int e) {
    if constexpr (LM == LD_EQ17) {
        const u64 q = lc.m.q;
#pragma unroll
        for (int k = 0; k < EL; ++k) x[k] = 0;
        for (int t = 0; t < lc.mu; ++t) {
            const Shoup g = lc.g[t];
            const u64 *bt = lc.b + (i64)t * lc.N + e;
#pragma unroll
            for (int k = 0; k < EL; ++k)
                x[k] = eq17_add<SMALL>(x[k], shoup_signed<Q1>(bt[k * DIST], g.w, g.wp, q), q);
        }
        if (lc.with_self) {
            const Shoup g = lc.g[lc.mu];
#pragma unroll
            for (int k = 0; k < EL; ++k)
                x[k] = eq17_sub<SMALL>(shoup_signed<Q1>(lc.a[e + k * DIST], g.w, g.wp, q), x[k], q);
        }
    } else if constexpr (LM == LD_SIGNED) {
        // all words first: one test says whether every sum is within the
        // product's range (|a|, |b| < 2^61, as errors and messages are), so the
        // reductions run side by side (a test per word: 14.5 us for a secret's
        // two limbs at N = 2^15)
        const u64 q = lc.m.q;
        const Shoup one = *lc.g;
        u64 out = 0;
#pragma unroll
        for (int k = 0; k < EL; ++k) {
            x[k] = lc.a[e + k * DIST];
            out |= x[k] + (1ull << 61);
        }
        if (lc.b) {
#pragma unroll
            for (int k = 0; k < EL; ++k) {
                const u64 y = lc.b[e + k * DIST];
                out |= y + (1ull << 61);
                x[k] += y;
            }
        }
        if ((out >> 62) == 0) {
#pragma unroll
            for (int k = 0; k < EL; ++k) {
                const u64 r = shoup_signed<Q1>(x[k], one.w, one.wp, q);
                x[k] = SMALL ? r : lift_sign(r, q);
            }
        } else {
#pragma unroll
            for (int k = 0; k < EL; ++k) x[k] = load_elem<LM, SMALL, Q1>(lc, e + k * DIST);
        }
    } else if constexpr (LM == LD_BCONVK) {
        constexpr int G = EL >= CKKS_NTT_MODDOWN_GROUP ? CKKS_NTT_MODDOWN_GROUP : EL;
#pragma unroll
        for (int k0 = 0; k0 < EL; k0 += G) {
            u64 r[G];
            scaled_bconv<G, DIST, Q1>(r, lc.b + e + k0 * DIST, lc.N, lc.cK, lc.K, lc.m);
#pragma unroll
            for (int u = 0; u < G; ++u) x[k0 + u] = r[u];
        }
    } else {
#pragma unroll
        for (int k = 0; k < EL; ++k) x[k] = load_elem<LM, SMALL, Q1>(lc, e + k * DIST);
    }
}

// Stores of one point set; the ModDown store takes four elements at a time,
// their K z-limb loads in flight together.
template <int EL, int DIST, int SM, bool FWD, bool SMALL, bool Q1>
__device__ __forceinline__ void store_set(const u64 (&x)[EL], const StoreCtx &sc, int e) {
    if constexpr (SM == ST_MODDOWN) {
        const u64 q = sc.m.q;
        constexpr int G = EL >= CKKS_NTT_MODDOWN_GROUP ? CKKS_NTT_MODDOWN_GROUP : EL;
#pragma unroll
        for (int k0 = 0; k0 < EL; k0 += G) {
            u64 r[G];
            scaled_bconv<G, DIST, Q1>(r, sc.aux + e + k0 * DIST, sc.N, sc.cK, sc.K, sc.m);
#pragma unroll
            for (int u = 0; u < G; ++u)
                sc.dst[e + (k0 + u) * DIST] = sub_mod(shoup_t<Q1>(x[k0 + u], sc.c.w, sc.c.wp, q), r[u], q);
        }
    } else {
#pragma unroll
        for (int k = 0; k < EL; ++k) store_elem<SM, SMALL, Q1>(sc, e + k * DIST, x[k], FWD);
    }
}

// Per-thread position in a phase: sub-problem and point-set lane.
struct Lane {
    u64 *sm;                 // the sub-problem's shared words (column: its column's)
    const ulonglong2 *tw;    // the sub-problem's twiddles (columns: the shared copy)
    int e;                   // element index of point 0
    int set;                 // point set of the first iteration
    int blk;                 // block within the warp (blocks only, else 0)
    bool active;
};

template <int LOGN, int LOGN2, bool FWD, int SH, int LM, int SM, bool SMALL, bool Q1, int I>
__device__ __forceinline__ void run_passes(const Lane &ln, u64 q, const LoadCtx &lc, const StoreCtx &sc) {
    constexpr int NP = Pass<LOGN, 0>::NP;
    if constexpr (I < NP) {
        typedef Geo<LOGN, LOGN2, SH> G;
        constexpr int P = FWD ? I : NP - 1 - I;
        constexpr int R = Pass<LOGN, P>::len, E0 = Pass<LOGN, P>::start, EL = 1 << R;
        constexpr bool first = I == 0, last = I == NP - 1;
        constexpr bool gin = first && LM >= 0 && PassAccess<LOGN, SH, P>::direct;
        constexpr bool gout = last && SM >= 0 && PassAccess<LOGN, SH, P>::direct;
        constexpr int t_min = G::n >> (E0 + R);
        constexpr int iters = (G::n >> R) / G::sets;
        u64 x[iters][EL];
        if constexpr (gin) {
            if (ln.active) {
#pragma unroll
                for (int it = 0; it < iters; ++it) {
                    const int set = ln.set + it * G::sets;
                    const int base = (set / t_min) * (G::n >> E0) + (set & (t_min - 1));
                    load_set<EL, t_min * G::stride, LM, SMALL, Q1>(x[it], lc, ln.e + base * G::stride);
                }
            }
        }
        // The data the previous pass exchanged is in place, and so are the
        // twiddles: of all columns (copied by the CTA; their copy was issued
        // before the loads above), or of this pass for the warp's blocks (the
        // I-th of NP groups).
        if constexpr (SH != COLS) async_wait<NP - 1 - I>();
        pass_sync<SH>();
        if (ln.active) {
#pragma unroll
            for (int it = 0; it < iters; ++it) {
                const int set = ln.set + it * G::sets;
                const int o = set & (t_min - 1), g = set / t_min;
                const int base = g * (G::n >> E0) + o;
                // columns: entry 0 unused; blocks: the warp's copy, passes in order of their stages
                const ulonglong2 *tw = ln.tw + (SH == COLS ? 1 << E0 : G::warp_blocks * ((1 << E0) - 1)) +
                                       ((ln.blk * (EL - 1)) << E0) + g;
                u64 *s = ln.sm + G::off(base);
                if constexpr (!gin) {
#pragma unroll
                    for (int k = 0; k < EL; ++k) x[it][k] = s[G::off(k * t_min)];
                }
                set_stages<R, E0, FWD, SMALL, Q1, (LOGN > 8)>(x[it], tw, q);
                // inverse: the output that is a sum at every stage (below
                // 288 q) -> [0, 2q); a store that multiplies takes it as it is
                if constexpr (!FWD && SMALL && !(gout && (SM == ST_SCALE || SM == ST_MODDOWN)))
                    x[it][0] = reduce_far(x[it][0] + (q << 9), q, lc.m.canon);
                if constexpr (gout) {
                    store_set<EL, t_min * G::stride, SM, FWD, SMALL, Q1>(x[it], sc, ln.e + base * G::stride);
                } else {
#pragma unroll
                    for (int k = 0; k < EL; ++k) s[G::off(k * t_min)] = x[it][k];
                }
            }
        }
        if constexpr (!gout && last) pass_sync<SH>();
        run_passes<LOGN, LOGN2, FWD, SH, LM, SM, SMALL, Q1, I + 1>(ln, q, lc, sc);
    }
}

// The twiddles of a warp's blocks, one commit group per pass in execution
// order: copied asynchronously while the data is loaded, so a warp waits for
// memory once instead of at every stage. (Read from L2 where they are used, the
// forward block phase had 6.4 of 12 stall cycles per issue on them.)
// The lanes (a warp's, or the CTA's for a whole limb) share the copies.
template <int LOGN, int LOGN2, bool FWD, int SH, int I>
__device__ __forceinline__ void copy_twiddles(ulonglong2 *dst, const ulonglong2 *tw, int N1, int b0, int lane) {
    constexpr int NP = Pass<LOGN, 0>::NP;
    if constexpr (I < NP) {
        typedef Geo<LOGN, LOGN2, SH> G;
        constexpr int T = SH == WHOLE ? G::sets : 32;
        constexpr int P = FWD ? I : NP - 1 - I;
        constexpr int R = Pass<LOGN, P>::len, E0 = Pass<LOGN, P>::start;
        constexpr int per = ((1 << R) - 1) << E0;  // entries per block
        ulonglong2 *d = dst + G::warp_blocks * ((1 << E0) - 1);
        const ulonglong2 *s = tw + ((i64)N1 << E0) + (i64)b0 * per;
        const int count = (N1 - b0 < G::warp_blocks ? N1 - b0 : G::warp_blocks) * per;
#pragma unroll
        for (int i = 0; i < (G::warp_blocks * per + T - 1) / T; ++i) {
            const int k = i * T + lane;
            if (k < count) async_copy16(d + k, s + k);
        }
        async_commit();
        copy_twiddles<LOGN, LOGN2, FWD, SH, I + 1>(dst, tw, N1, b0, lane);
    }
}

// One tile (CTA) of one limb: tile index `tile` of the phase.
template <int LOGN, int LOGN2, bool FWD, int SH, int LM, int SM, bool SMALL, bool Q1>
__device__ __forceinline__ void phase_tile(u64 *sm, const NttPhase &P, const ulonglong2 *tw, u64 q,
                                           const LoadCtx &lc, const StoreCtx &sc, int tile) {
    typedef Geo<LOGN, LOGN2, SH> G;
    constexpr int n = G::n, NP = Pass<LOGN, 0>::NP;
    const int tid = threadIdx.x;
    Lane ln;
    if constexpr (SH == COLS) {
        const int groups = blockDim.x / G::group;
        const int grp = tid / G::group;
        ulonglong2 *tws = reinterpret_cast<ulonglong2 *>(sm + groups * G::unit);
        ln.sm = sm + grp * G::unit + (tid & 15);
        ln.tw = tws;
        ln.e = (tile * groups + grp) * 16 + (tid & 15);
        ln.set = (tid / 16) % G::sets;
        ln.blk = 0;
        ln.active = true;
        // the n - 1 twiddles every column shares, copied while the first
        // pass's loads are in flight
        for (int i = tid; i < n; i += blockDim.x) tws[i] = tw[i];
        grid_dependency_wait();
        run_passes<LOGN, LOGN2, FWD, SH, LM, SM, SMALL, Q1, 0>(ln, q, lc, sc);
    } else {
        // a warp and its blocks, or the CTA and its limb
        constexpr int BW = G::warp_blocks;
        constexpr int T = SH == WHOLE ? G::sets : 32;
        constexpr int W = (BW * n + T - 1) / T;           // words per lane
        constexpr int U = W < 8 ? W : 8;
        constexpr int PF = FWD ? 0 : NP - 1, PL = FWD ? NP - 1 : 0;
        // a limb of N <= 2^8 may be less than a word per lane, or a set
        constexpr bool FULL = LOGN2 != 0 || SH == WHOLE;
        const int lane = SH == WHOLE ? tid : tid & 31;
        const int b0 = !FULL || SH == WHOLE ? 0 : tile * (blockDim.x / G::sets) + (tid / 32) * BW;  // first block in the limb
        u64 *wsm = SH == WHOLE ? sm : reinterpret_cast<u64 *>(reinterpret_cast<char *>(sm) + (tid / 32) * G::warp_bytes);
        ulonglong2 *wtw = reinterpret_cast<ulonglong2 *>(wsm + G::warp_data);
        ln.blk = SH == WHOLE ? 0 : lane / G::sets;
        ln.sm = wsm + ln.blk * G::unit;
        ln.tw = wtw;
        ln.set = SH == WHOLE ? lane : lane % G::sets;
        ln.e = (b0 + ln.blk) << LOGN;
        ln.active = FULL || b0 + ln.blk < P.N1;
        copy_twiddles<LOGN, LOGN2, FWD, SH, 0>(wtw, tw, P.N1, b0, lane);
        grid_dependency_wait();
        const int words = (P.N1 - b0) * n;                // words of the limb from the first block on
        const int e0 = b0 << LOGN;
        // shared offset of word idx of the warp's blocks
        auto woff = [](int idx) { return (idx >> LOGN) * G::unit + G::off(idx & (n - 1)); };
        // run-time modes (N <= 2^8): both sides staged, one element at a time
        constexpr bool RT = LM < 0;
        if constexpr (RT) {
#pragma unroll 1
            for (int idx = lane; idx < W * T; idx += T)
                if (idx < words) wsm[woff(idx)] = load_elem<LM, SMALL, Q1>(lc, e0 + idx);
        } else if constexpr (!PassAccess<LOGN, SH, PF>::direct) {
            // coalesced global -> shared with the fused load, U loads in flight
#pragma unroll
            for (int i0 = 0; i0 < W; i0 += U) {
                u64 v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int idx = lane + T * (i0 + u);
                    if (FULL || idx < words) v[u] = load_elem<LM, SMALL, Q1>(lc, e0 + idx);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int idx = lane + T * (i0 + u);
                    if (FULL || idx < words) wsm[woff(idx)] = v[u];
                }
            }
        }
        run_passes<LOGN, LOGN2, FWD, SH, LM, SM, SMALL, Q1, 0>(ln, q, lc, sc);
        if constexpr (RT) {
#pragma unroll 1
            for (int idx = lane; idx < W * T; idx += T)
                if (idx < words) store_elem<SM, SMALL, Q1>(sc, e0 + idx, wsm[woff(idx)], FWD);
        } else if constexpr (!PassAccess<LOGN, SH, PL>::direct) {
            // shared -> global with the fused store (coalesced); a store that
            // reads an aux limb gathers U elements and their aux words first
#pragma unroll
            for (int i0 = 0; i0 < W; i0 += U) {
                if constexpr (SM == ST_MRS || SM == ST_ADDSUB) {
                    u64 a[U], a2[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int idx = lane + T * (i0 + u);
                        if (FULL || idx < words) {
                            a[u] = sc.aux[e0 + idx];
                            if (SM == ST_ADDSUB) a2[u] = sc.aux2[e0 + idx];
                        }
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int idx = lane + T * (i0 + u);
                        if (FULL || idx < words) {
                            const u64 r = canonical<SMALL>(wsm[woff(idx)], q, sc.m.canon);
                            if (SM == ST_MRS)
                                sc.dst[e0 + idx] = sub_mod(shoup_t<Q1>(a[u], sc.c.w, sc.c.wp, q), r, q);
                            else sc.dst[e0 + idx] = sub_mod(add_mod(a[u], a2[u], q), r, q);
                        }
                    }
                } else {
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int idx = lane + T * (i0 + u);
                        if (FULL || idx < words) store_elem<SM, SMALL, Q1>(sc, e0 + idx, wsm[woff(idx)], FWD);
                    }
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------
// the phase kernels: grid (tiles, limbs) for uniform launches, one
// flattened dimension (limb * tiles + tile) for table launches
// ---------------------------------------------------------------------------
template <int LOGN, int LOGN2, bool FWD, int SH, int LM, int SM, int MINB, bool Q1>
__global__ void __launch_bounds__(kPhaseThreads, MINB) ntt_phase_kernel(NttPhase P, LimbJobs J, LoadSpec L, StoreSpec S) {
    extern __shared__ __align__(16) u64 sm[];
    int b, p, l, job = blockIdx.y;
    if constexpr (SH == BLOCKS && LOGN2 == 0) {  // N <= 2^8: a limb per warp
        job = job * (blockDim.x / 32) + threadIdx.x / 32;
        if (job >= J.n_batch * J.n_polys * J.n_limbs) return;
    }
    decode_job(J, job, b, p, l);
    const int prime = J.prime[l];
    const ModQ m = P.mods[prime];
    const ulonglong2 *tw = (FWD ? P.tw_fwd : P.tw_inv) + (i64)prime * P.N;
    const LoadCtx lc = make_load(L, J, P.N, b, p, l, prime, m);
    const StoreCtx sc = make_store(S, J, P.N, b, p, l, prime, m);
    if (small_prime(m.q)) phase_tile<LOGN, LOGN2, FWD, SH, LM, SM, true, Q1>(sm, P, tw, m.q, lc, sc, blockIdx.x);
    else phase_tile<LOGN, LOGN2, FWD, SH, LM, SM, false, Q1>(sm, P, tw, m.q, lc, sc, blockIdx.x);
}

template <int LOGN, int LOGN2, bool FWD, int SH, int LM, int SM, int MINB, bool Q1>
__global__ void __launch_bounds__(kPhaseThreads, MINB) ntt_phase_table_kernel(NttPhase P, const NttJob *jobs, int tiles,
                                                                    LoadSpec L, StoreSpec S) {
    extern __shared__ __align__(16) u64 sm[];
    grid_dependency_wait();  // the job table may have been written just before
    const int job = blockIdx.x / tiles;
    const int tile = blockIdx.x - job * tiles;
    const NttJob j = jobs[job];
    const ModQ m = P.mods[j.prime];
    const ulonglong2 *tw = (FWD ? P.tw_fwd : P.tw_inv) + (i64)j.prime * P.N;
    const LoadCtx lc = make_load(L, j, P.N, m);
    const StoreCtx sc = make_store(S, j, P.N, m);
    if (small_prime(m.q)) phase_tile<LOGN, LOGN2, FWD, SH, LM, SM, true, Q1>(sm, P, tw, m.q, lc, sc, tile);
    else phase_tile<LOGN, LOGN2, FWD, SH, LM, SM, false, Q1>(sm, P, tw, m.q, lc, sc, tile);
}

// ---------------------------------------------------------------------------
// host-side launch of one instantiation
// ---------------------------------------------------------------------------
struct PhaseLaunch {
    PhaseShape s;
    cudaStream_t st;
};

// Resident CTAs of 256 threads per SM the kernels are compiled for.
#ifndef CKKS_NTT_COL_MINB
#define CKKS_NTT_COL_MINB 4     // columns: 64 registers (871 vs 842 G butterflies/s with three CTAs, 736 with two)
#endif
#ifndef CKKS_NTT_COL_WIDE_MINB
#define CKKS_NTT_COL_WIDE_MINB 4  // columns with an Eq. 17 load (411 -> 393 us per k = 12, batch 8 launch
                                  // against three CTAs)
#endif
#ifndef CKKS_NTT_COL_MODDOWN_MINB
#define CKKS_NTT_COL_MODDOWN_MINB 3  // columns with a signed load or a store that sums over the K z-limbs: 80 registers
#endif
#ifndef CKKS_NTT_COL_BCONVK_MINB
#define CKKS_NTT_COL_BCONVK_MINB 2  // columns whose load sums over the K z-limbs: 128 registers
#endif
#ifndef CKKS_NTT_BLOCK_MINB
#define CKKS_NTT_BLOCK_MINB 2   // blocks: shared memory holds the twiddles of 16 warps per SM
#endif

template <typename K>
static inline cudaError_t allow_smem(K kern, size_t smem) {
    if (smem > 48 * 1024) return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    return cudaSuccess;
}

template <int LOGN, int LOGN2, bool FWD, int SH, int LM, int SM, int MINB, bool Q1>
static inline cudaError_t launch_uniform(const NttPhase &P, const LimbJobs &J, const LoadSpec &L,
                                         const StoreSpec &S, const PhaseLaunch &G) {
    auto kern = ntt_phase_kernel<LOGN, LOGN2, FWD, SH, LM, SM, MINB, Q1>;
    cudaError_t e = allow_smem(kern, G.s.smem);
    if (e != cudaSuccess) return e;
    const int limbs = J.n_batch * J.n_polys * J.n_limbs;
    if (limbs > 65535) return cudaErrorInvalidConfiguration;  // the grid's second dimension, one limb each
    dim3 grid(G.s.tiles, (limbs + G.s.limbs - 1) / G.s.limbs);
    return launch_dependent(kern, grid, dim3(G.s.threads), G.s.smem, G.st, P, J, L, S);
}

template <int LOGN, int LOGN2, bool FWD, int SH, int LM, int SM, int MINB, bool Q1>
static inline cudaError_t launch_table(const NttPhase &P, const NttJob *jobs, int n_jobs, const LoadSpec &L,
                                       const StoreSpec &S, const PhaseLaunch &G) {
    auto kern = ntt_phase_table_kernel<LOGN, LOGN2, FWD, SH, LM, SM, MINB, Q1>;
    cudaError_t e = allow_smem(kern, G.s.smem);
    if (e != cudaSuccess) return e;
    const long long blocks = (long long)n_jobs * G.s.tiles;
    if (blocks <= 0) return cudaSuccess;
    if (blocks > 0x7FFFFFFFll) return cudaErrorInvalidValue;
    return launch_dependent(kern, dim3((unsigned)blocks), dim3(G.s.threads), G.s.smem, G.st, P, jobs, G.s.tiles, L, S);
}

// Dispatch of one direction (FWD) and job source (TABLE) over the shape, log2
// n and the modes. Every pair of modes the library uses has its own kernel, for
// tables those that waves use (a kernel with run-time modes kept every mode's pointers alive and its code
// did not fit the instruction cache: 12-18 us a launch at N = 2^10 against
// 5-7): a phase that fuses a mode has the plain mode on its other side.
//   two phases (N >= 2^13): dispatch_two, with the products in the form Q1
//   selects (N >= 2^14);
//   one phase (2^9 <= N <= 2^12): dispatch_whole;
//   N <= 2^8: dispatch_tiny, the plain transforms with a kernel of their own,
//   the others run-time modes.
#define CKKS_LAUNCH(LG, LG2, SHv, LMv, SMv, MB, Q)                                                   \
    do {                                                                                             \
        if constexpr (TABLE) return launch_table<LG, LG2, FWD, SHv, LMv, SMv, MB, Q>(P, jobs, n_jobs, L, S, G); \
        else return launch_uniform<LG, LG2, FWD, SHv, LMv, SMv, MB, Q>(P, *J, L, S, G);              \
    } while (0)
#define CKKS_MODES(LMv, SMv) if (L.mode == LMv && S.mode == SMv)

template <bool FWD, bool TABLE, bool Q1, int LG, int LG2>
static inline cudaError_t dispatch_cols(const NttPhase &P, const LimbJobs *J, const NttJob *jobs, int n_jobs,
                                        const LoadSpec &L, const StoreSpec &S, const PhaseLaunch &G) {
    if constexpr (FWD) {
        CKKS_MODES(LD_PLAIN, ST_LAZY) CKKS_LAUNCH(LG, LG2, COLS, LD_PLAIN, ST_LAZY, CKKS_NTT_COL_MINB, Q1);
        CKKS_MODES(LD_EQ17, ST_LAZY) CKKS_LAUNCH(LG, LG2, COLS, LD_EQ17, ST_LAZY, CKKS_NTT_COL_WIDE_MINB, Q1);
        if constexpr (!TABLE) {
            CKKS_MODES(LD_BCONVK, ST_LAZY) CKKS_LAUNCH(LG, LG2, COLS, LD_BCONVK, ST_LAZY, CKKS_NTT_COL_BCONVK_MINB, Q1);
            CKKS_MODES(LD_SIGNED, ST_LAZY) CKKS_LAUNCH(LG, LG2, COLS, LD_SIGNED, ST_LAZY, CKKS_NTT_COL_MODDOWN_MINB, Q1);
        }
    } else {
        CKKS_MODES(LD_PLAIN, ST_SCALE) CKKS_LAUNCH(LG, LG2, COLS, LD_PLAIN, ST_SCALE, CKKS_NTT_COL_MINB, Q1);
        CKKS_MODES(LD_PLAIN, ST_MODDOWN) CKKS_LAUNCH(LG, LG2, COLS, LD_PLAIN, ST_MODDOWN, CKKS_NTT_COL_MODDOWN_MINB, Q1);
    }
    return cudaErrorInvalidValue;
}

template <bool FWD, bool TABLE, bool Q1, int LG>
static inline cudaError_t dispatch_blocks(const NttPhase &P, const LimbJobs *J, const NttJob *jobs, int n_jobs,
                                          const LoadSpec &L, const StoreSpec &S, const PhaseLaunch &G) {
    if constexpr (FWD) {
        CKKS_MODES(LD_PLAIN, ST_REDUCE) CKKS_LAUNCH(LG, LG, BLOCKS, LD_PLAIN, ST_REDUCE, CKKS_NTT_BLOCK_MINB, Q1);
        CKKS_MODES(LD_PLAIN, ST_MRS) CKKS_LAUNCH(LG, LG, BLOCKS, LD_PLAIN, ST_MRS, CKKS_NTT_BLOCK_MINB, Q1);
        if constexpr (!TABLE)
            CKKS_MODES(LD_PLAIN, ST_ADDSUB) CKKS_LAUNCH(LG, LG, BLOCKS, LD_PLAIN, ST_ADDSUB, CKKS_NTT_BLOCK_MINB, Q1);
    } else {
        CKKS_MODES(LD_PLAIN, ST_LAZY) CKKS_LAUNCH(LG, LG, BLOCKS, LD_PLAIN, ST_LAZY, CKKS_NTT_BLOCK_MINB, Q1);
        CKKS_MODES(LD_ADD, ST_LAZY) CKKS_LAUNCH(LG, LG, BLOCKS, LD_ADD, ST_LAZY, CKKS_NTT_BLOCK_MINB, Q1);
    }
    return cudaErrorInvalidValue;
}

template <bool FWD, bool TABLE, bool Q1>
static inline cudaError_t dispatch_two(int logn, const NttPhase &P, const LimbJobs *J, const NttJob *jobs,
                                       int n_jobs, const LoadSpec &L, const StoreSpec &S, const PhaseLaunch &G) {
#define CKKS_COLS(LG, LG2) \
    if (logn == LG && P.log_n2 == LG2) return dispatch_cols<FWD, TABLE, Q1, LG, LG2>(P, J, jobs, n_jobs, L, S, G)
    if (G.s.shape == COLS) {
        if constexpr (!Q1) CKKS_COLS(6, 7);
        CKKS_COLS(7, 7);
        CKKS_COLS(7, 8);
        CKKS_COLS(8, 8);
    } else {
        if (logn == 7) return dispatch_blocks<FWD, TABLE, Q1, 7>(P, J, jobs, n_jobs, L, S, G);
        if (logn == 8) return dispatch_blocks<FWD, TABLE, Q1, 8>(P, J, jobs, n_jobs, L, S, G);
    }
#undef CKKS_COLS
    return cudaErrorInvalidValue;
}

template <bool FWD, bool TABLE, int LG>
static inline cudaError_t dispatch_whole_n(const NttPhase &P, const LimbJobs *J, const NttJob *jobs, int n_jobs,
                                           const LoadSpec &L, const StoreSpec &S, const PhaseLaunch &G) {
    if constexpr (FWD) {
        CKKS_MODES(LD_PLAIN, ST_REDUCE) CKKS_LAUNCH(LG, 0, WHOLE, LD_PLAIN, ST_REDUCE, 2, false);
        if constexpr (!TABLE)
            CKKS_MODES(LD_SIGNED, ST_REDUCE) CKKS_LAUNCH(LG, 0, WHOLE, LD_SIGNED, ST_REDUCE, 2, false);
        CKKS_MODES(LD_EQ17, ST_REDUCE) CKKS_LAUNCH(LG, 0, WHOLE, LD_EQ17, ST_REDUCE, 2, false);
        CKKS_MODES(LD_EQ17, ST_MRS) CKKS_LAUNCH(LG, 0, WHOLE, LD_EQ17, ST_MRS, 2, false);
        if constexpr (!TABLE) {
            CKKS_MODES(LD_BCONVK, ST_ADDSUB) CKKS_LAUNCH(LG, 0, WHOLE, LD_BCONVK, ST_ADDSUB, 2, false);
            CKKS_MODES(LD_PLAIN, ST_ADDSUB) CKKS_LAUNCH(LG, 0, WHOLE, LD_PLAIN, ST_ADDSUB, 2, false);
        }
    } else {
        CKKS_MODES(LD_PLAIN, ST_SCALE) CKKS_LAUNCH(LG, 0, WHOLE, LD_PLAIN, ST_SCALE, 2, false);
        CKKS_MODES(LD_ADD, ST_MODDOWN) CKKS_LAUNCH(LG, 0, WHOLE, LD_ADD, ST_MODDOWN, 2, false);
        if constexpr (!TABLE)
            CKKS_MODES(LD_PLAIN, ST_MODDOWN) CKKS_LAUNCH(LG, 0, WHOLE, LD_PLAIN, ST_MODDOWN, 2, false);
    }
    return cudaErrorInvalidValue;
}

template <bool FWD, bool TABLE>
static inline cudaError_t dispatch_whole(int logn, const NttPhase &P, const LimbJobs *J, const NttJob *jobs,
                                         int n_jobs, const LoadSpec &L, const StoreSpec &S, const PhaseLaunch &G) {
    switch (logn) {
    case 9: return dispatch_whole_n<FWD, TABLE, 9>(P, J, jobs, n_jobs, L, S, G);
    case 10: return dispatch_whole_n<FWD, TABLE, 10>(P, J, jobs, n_jobs, L, S, G);
    case 11: return dispatch_whole_n<FWD, TABLE, 11>(P, J, jobs, n_jobs, L, S, G);
    case 12: return dispatch_whole_n<FWD, TABLE, 12>(P, J, jobs, n_jobs, L, S, G);
    default: return cudaErrorInvalidValue;
    }
}

template <bool FWD>
static inline cudaError_t dispatch_tiny(int logn, const NttPhase &P, const LimbJobs *J, const LoadSpec &L,
                                        const StoreSpec &S, const PhaseLaunch &G) {
    constexpr bool TABLE = false;
    const NttJob *jobs = nullptr;
    const int n_jobs = 0;
#define CKKS_TINY(LG)                                                                             \
    case LG:                                                                                      \
        if constexpr (FWD) {                                                                      \
            CKKS_MODES(LD_PLAIN, ST_REDUCE) CKKS_LAUNCH(LG, 0, BLOCKS, LD_PLAIN, ST_REDUCE, 2, false); \
        } else {                                                                                  \
            CKKS_MODES(LD_PLAIN, ST_SCALE) CKKS_LAUNCH(LG, 0, BLOCKS, LD_PLAIN, ST_SCALE, 2, false); \
        }                                                                                         \
        CKKS_LAUNCH(LG, 0, BLOCKS, -1, -1, 2, false)
    switch (logn) {
        CKKS_TINY(4);
        CKKS_TINY(5);
        CKKS_TINY(6);
        CKKS_TINY(7);
        CKKS_TINY(8);
    default: return cudaErrorInvalidValue;
    }
#undef CKKS_TINY
}
#undef CKKS_LAUNCH
#undef CKKS_MODES

// One translation unit per direction, job source (u: uniform, t: table) and
// product form (ntt_*1.cu: primes = 1 (mod 2^32)) so that they compile in
// parallel; ntt_whole_*.cu hold the one-phase kernels.
#define CKKS_DECL(name)                                                                              \
    cudaError_t name(int logn, const NttPhase &P, const LimbJobs *J, const NttJob *jobs, int n_jobs, \
                     const LoadSpec &L, const StoreSpec &S, const PhaseLaunch &G)
CKKS_DECL(ntt_two_uf);
CKKS_DECL(ntt_two_ui);
CKKS_DECL(ntt_two_tf);
CKKS_DECL(ntt_two_ti);
CKKS_DECL(ntt_two_uf1);
CKKS_DECL(ntt_two_ui1);
CKKS_DECL(ntt_two_tf1);
CKKS_DECL(ntt_two_ti1);
CKKS_DECL(ntt_whole_uf);
CKKS_DECL(ntt_whole_ui);
CKKS_DECL(ntt_whole_tf);
CKKS_DECL(ntt_whole_ti);
#undef CKKS_DECL

}  // namespace ckks
