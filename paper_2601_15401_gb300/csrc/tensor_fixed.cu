// Tensor products (Eq. 1, 8, 13) of tree nodes in fixed shapes.
//
// The tensor kernels of rns.cu unroll their product loops to a tuple-size
// bound and predicate every product on the run-time tuple sizes: a node of
// two 7-term tuples issues the instructions of 91 products for its 49. The
// kernels here are compiled for one node shape each: children sorted by
// size, largest first (the product is commutative and every step returns
// canonical residues, so the order does not change the result), every load
// of the node issued before the first product, each output term stored as
// soon as it is reduced. Shapes (kTensorShapes): two children of 4..7
// terms, three of 4 or 5 terms — among them the roots and the larger inner
// nodes of the paper's partitions for k = 6..12 (Table II) — and, on limbs,
// the small nodes: two or three ciphertexts, two children of 3 terms, alone or
// with a ciphertext.
//
// Operands are reduced residues and no term sums more than 7 products, so
// the 128-bit sums need no per-term reduction: B q^2 < q 2^64 for B <= 8
// and q < 2^61 keeps the high word below q, as REDC requires. With every
// prime below 2^60 (LIMB) the products run on 30-bit limbs (DotLimbs, at most
// 8 terms): three multiply-adds each.
#include <utility>

#include "common.cuh"
#include "internal.h"
#include "rns.h"

namespace ckks {

namespace {

constexpr int kThreads = 256;

// CTAs per SM a shape is compiled for: four for two 4-term children on limbs,
// three for all others (three ciphertexts on limbs: 118.6 us with three, 121
// with four; two 4-term children as 128-bit products, 24 limbs at N = 2^16:
// 43.1 us with three, 44.0 with four).
template <int A, int B, int C, bool LIMB>
constexpr int kFixedMinb = LIMB && A > 3 && A + B + C <= 8 ? 4 : 3;

// A residue as an operand of the dot products, itself or its limbs, and the
// reduction of a sum of at most 8 products of residues. (The sums of limbs
// are put together as 128-bit words for the REDC: reducing them by limbs, as
// BConv does, took 155 against 137 us for two 4-term children, the final
// subtractions costing more than the multiplies saved.)
template <bool LIMB, bool Q1>
struct Operand {
    typedef u64 type;
    typedef Acc128Lazy acc;
    static __device__ __forceinline__ u64 make(u64 v) { return v; }
    static __device__ __forceinline__ u64 reduce(const Acc128Lazy &a, const ModQ &m) { return redc_t<Q1>(a.hi, a.lo, m); }
};
template <bool Q1>
struct Operand<true, Q1> {
    typedef Limbs type;
    typedef DotLimbs acc;
    static __device__ __forceinline__ Limbs make(u64 v) { return split_limbs<30>(v); }
    static __device__ __forceinline__ u64 reduce(const DotLimbs &a, const ModQ &m) {
        u64 hi, lo;
        a.value<30>(hi, lo);
        return redc_t<Q1>(hi, lo, m);
    }
};

// term t of x * y (polynomials in s of A and B terms) at coefficient e, reduced
template <int A, int B, int V, bool Q1, bool LIMB>
__device__ __forceinline__ u64 conv_term(const typename Operand<LIMB, Q1>::type (&x)[A][V],
                                         const typename Operand<LIMB, Q1>::type (&y)[B][V], int t, int e,
                                         const ModQ m) {
    static_assert(A >= B && B <= 8, "at most 8 products per term");
    typename Operand<LIMB, Q1>::acc acc;
    acc.zero();
#pragma unroll
    for (int b = 0; b < B; ++b)
        if (t - b >= 0 && t - b < A) acc.mac(x[t - b][e], y[b][e]);
    return Operand<LIMB, Q1>::reduce(acc, m);
}

template <int T, int V>
__device__ __forceinline__ void load_terms(const u64 *src, i64 ps, u64 (&o)[T][V]) {
#pragma unroll
    for (int a = 0; a < T; ++a) load_span<V>(src + (i64)a * ps, o[a]);
}

// V adjacent coefficients r (= limb j * N + coefficient) of a node with
// children of A, B (and C; 0 for two children) terms: m - 1 Montgomery
// products, which leave R^-(m-1), and R^(m-1) as a Shoup product by a per-prime
// constant on the terms of the last child.
template <int A, int B, int C, int V, bool Q1, bool LIMB, class View>
__device__ __forceinline__ void tensor_fixed_coeff(const View &v, i64 r, int j, const ModQ m, const Shoup *rfix) {
    typedef Operand<LIMB, Q1> Op;
    const Shoup fix = rfix[(i64)j * 16 + (C ? 3 : 2)];
    constexpr int Z = A + B - 1, CC = C ? C : 1;
    u64 x[A][V], y[B][V], w[CC][V];
    load_terms<A, V>(v.src(0) + r, v.pstride(0), x);
    load_terms<B, V>(v.src(1) + r, v.pstride(1), y);
    if constexpr (C != 0) load_terms<C, V>(v.src(2) + r, v.pstride(2), w);
    u64 *dst = v.dst() + r;
    const i64 ds = v.dstride();
    typename Op::type xo[A][V], yo[B][V];
#pragma unroll
    for (int e = 0; e < V; ++e) {
#pragma unroll
        for (int a = 0; a < A; ++a) xo[a][e] = Op::make(x[a][e]);
#pragma unroll
        for (int b = 0; b < B; ++b)
            yo[b][e] = Op::make(C ? y[b][e] : shoup_t<Q1>(y[b][e], fix.w, fix.wp, m.q));
    }
    if constexpr (C == 0) {
#pragma unroll
        for (int t = 0; t < Z; ++t) {
            u64 o[V];
#pragma unroll
            for (int e = 0; e < V; ++e) o[e] = conv_term<A, B, V, Q1, LIMB>(xo, yo, t, e, m);
            store_span<V>(dst + (i64)t * ds, o);
        }
    } else {
        typename Op::type zo[Z][V], wo[CC][V];
#pragma unroll
        for (int e = 0; e < V; ++e) {
#pragma unroll
            for (int t = 0; t < Z; ++t) zo[t][e] = Op::make(conv_term<A, B, V, Q1, LIMB>(xo, yo, t, e, m));
#pragma unroll
            for (int a = 0; a < CC; ++a) wo[a][e] = Op::make(shoup_t<Q1>(w[a][e], fix.w, fix.wp, m.q));
        }
#pragma unroll
        for (int t = 0; t < Z + CC - 1; ++t) {
            u64 o[V];
#pragma unroll
            for (int e = 0; e < V; ++e) o[e] = conv_term<Z, CC, V, Q1, LIMB>(zo, wo, t, e, m);
            store_span<V>(dst + (i64)t * ds, o);
        }
    }
}

template <int A, int B, int C, int V, bool Q1, bool LIMB>
__global__ void __launch_bounds__(kThreads, kFixedMinb<A, B, C, LIMB>) tensor_fixed_kernel(TensorArgs T) {
    grid_dependency_wait();
    const i64 r = ((i64)blockIdx.x * blockDim.x + threadIdx.x) * V;  // limb * N + coefficient
    if (r >= (i64)T.level * T.N) return;
    const int j = (int)(r >> T.log_n);
    tensor_fixed_coeff<A, B, C, V, Q1, LIMB>(TensorUniformView{T, (int)blockIdx.y}, r, j, T.mods[j], T.rfix);
}

// blockIdx.y = table entry (every entry of the launch has this shape); the
// entry is staged in shared memory, one word per thread
template <int A, int B, int C, int V, bool Q1, bool LIMB>
__global__ void __launch_bounds__(kThreads, kFixedMinb<A, B, C, LIMB>) tensor_fixed_table_kernel(const TensorJob *jobs, int N, int log_n,
                                                                        const ModQ *mods, const Shoup *rfix) {
    grid_dependency_wait();
    __shared__ TensorJob J;
    {
        static_assert(sizeof(TensorJob) % sizeof(u64) == 0, "TensorJob is a whole number of words");
        constexpr int W = sizeof(TensorJob) / sizeof(u64);
        const u64 *src = reinterpret_cast<const u64 *>(jobs + blockIdx.y);
        u64 *dst = reinterpret_cast<u64 *>(&J);
        for (int i = threadIdx.x; i < W; i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
    const i64 r = ((i64)blockIdx.x * blockDim.x + threadIdx.x) * V;
    if (r >= (i64)J.level * N) return;
    const int j = (int)(r >> log_n);
    tensor_fixed_coeff<A, B, C, V, Q1, LIMB>(TensorTableView{J}, r, j, mods[j], rfix);
}

// f(A, B, C) with the shape of `code` (kTensorShapes) as integral constants
template <int I = 0, class F>
cudaError_t with_shape(int code, F &&f) {
    if constexpr (I < kTensorShapeCount) {
        if (code == I)
            return f(std::integral_constant<int, kTensorShapes[I].a>{}, std::integral_constant<int, kTensorShapes[I].b>{},
                     std::integral_constant<int, kTensorShapes[I].c>{});
        return with_shape<I + 1>(code, f);
    } else {
        return cudaErrorInvalidValue;
    }
}

// Small tuples (up to 3 terms a child; only on limbs) take two adjacent
// coefficients per thread where every pointer allows 16-byte accesses.
template <int A, bool LIMB>
constexpr bool kSmallShape = A <= 3 && LIMB;

template <bool Q1, bool LIMB>
cudaError_t launch_uniform(const TensorArgs &T, int code, bool vec2, cudaStream_t st) {
    return with_shape(code, [&](auto a, auto b, auto c) {
        constexpr int A = decltype(a)::value, B = decltype(b)::value, C = decltype(c)::value;
        auto go = [&](auto kern, int V) {
            const i64 per = (i64)kThreads * V;
            dim3 blocks((unsigned)(((i64)T.level * T.N + per - 1) / per), T.n_batch);
            return launch_dependent(kern, blocks, dim3(kThreads), 0, st, T);
        };
        if constexpr (A <= 3 && !LIMB) return cudaErrorInvalidValue;
        else {
            if constexpr (kSmallShape<A, LIMB>)
                if (vec2) return go(tensor_fixed_kernel<A, B, C, 2, Q1, LIMB>, 2);
            return go(tensor_fixed_kernel<A, B, C, 1, Q1, LIMB>, 1);
        }
    });
}

template <bool Q1, bool LIMB>
cudaError_t launch_table(const Context &C_, const TensorJob *jobs, int n_jobs, int code, int max_level, bool vec2,
                         cudaStream_t st) {
    return with_shape(code, [&](auto a, auto b, auto c) {
        constexpr int A = decltype(a)::value, B = decltype(b)::value, C = decltype(c)::value;
        auto go = [&](auto kern, int V) {
            const i64 per = (i64)kThreads * V;
            dim3 blocks((unsigned)(((i64)max_level * C_.N + per - 1) / per), (unsigned)n_jobs);
            return launch_dependent(kern, blocks, dim3(kThreads), 0, st, jobs, C_.N, C_.log_n, C_.d_mods, C_.d_rfix);
        };
        if constexpr (A <= 3 && !LIMB) return cudaErrorInvalidValue;
        else {
            if constexpr (kSmallShape<A, LIMB>)
                if (vec2) return go(tensor_fixed_table_kernel<A, B, C, 2, Q1, LIMB>, 2);
            return go(tensor_fixed_table_kernel<A, B, C, 1, Q1, LIMB>, 1);
        }
    });
}

}  // namespace

int tensor_sort_children(TensorJob &T) {
    for (int c = 1; c < T.m; ++c)
        for (int d = c; d > 0 && T.cpolys[d] > T.cpolys[d - 1]; --d) {
            std::swap(T.child[d], T.child[d - 1]);
            std::swap(T.cstride[d], T.cstride[d - 1]);
            std::swap(T.cpolys[d], T.cpolys[d - 1]);
        }
    if (T.m < 2 || T.m > 3) return -1;
    return tensor_fixed_code(T.m, T.cpolys[0], T.cpolys[1], T.m > 2 ? T.cpolys[2] : 0);
}

int tensor_sort_children(TensorArgs &A) {
    for (int c = 1; c < A.m; ++c)
        for (int d = c; d > 0 && A.child_polys[d] > A.child_polys[d - 1]; --d) {
            std::swap(A.child[d], A.child[d - 1]);
            std::swap(A.child_polys[d], A.child_polys[d - 1]);
        }
    if (A.m < 2 || A.m > 3) return -1;
    return tensor_fixed_code(A.m, A.child_polys[0], A.child_polys[1], A.m > 2 ? A.child_polys[2] : 0);
}

cudaError_t launch_tensor_fixed(const Context &C, const TensorArgs &A, int code, bool vec2, cudaStream_t st) {
    return with_product_form(C, [&](auto q1, auto limb) {
        return launch_uniform<q1.value, limb.value>(A, code, vec2, st);
    });
}

cudaError_t launch_tensor_fixed_table(const Context &C, const TensorJob *jobs, int n_jobs, int code, int max_level,
                                      bool vec2, double bytes, double ops, cudaStream_t st) {
    if (n_jobs <= 0) return cudaSuccess;
    if (n_jobs > 65535) return cudaErrorInvalidValue;
    count_kernel(C);
    ProfScope ps(C, KC_TENSOR, bytes, st, ops);
    return with_product_form(C, [&](auto q1, auto limb) {
        return launch_table<q1.value, limb.value>(C, jobs, n_jobs, code, max_level, vec2, st);
    });
}

}  // namespace ckks
