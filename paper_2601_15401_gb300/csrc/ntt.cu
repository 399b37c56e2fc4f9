// Host side of the negacyclic NTT / INTT (the kernels and their design are
// described in ntt_kernel.cuh): phase geometry, algorithmic byte and Shoup
// product counts for the timing hook, and the two-phase transform with fused
// first load / last store.
#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "ntt_kernel.cuh"

namespace ckks {

// Table position of forward / inverse twiddle k (psi^(+-)brv(k)) in the order
// the passes read it (ntt_kernel.cuh): k = m_glob + i, m_glob = 2^s, is stage s
// of the transform; its first log_n1 stages run in the column phase, the
// others in the block phase, in passes of up to CKKS_NTT_RMAX stages.
int twiddle_slot(int logN, int k) {
    if (k == 0) return 0;
    int log_n1, log_n2;
    ntt_geometry(logN, log_n1, log_n2);
    int s = 0;
    while ((k >> (s + 1)) != 0) ++s;
    const bool cols = s < log_n1;
    const int logn = cols ? log_n1 : log_n2;
    const int ls = cols ? s : s - log_n1;          // stage within the phase
    const int m_loc = 1 << ls;
    const int i = cols ? k - m_loc : k & (m_loc - 1);  // group within the sub-problem
    const int b = cols ? 0 : (k >> ls) - (1 << log_n1);  // k = m_loc (N1 + b) + i
    // the pass of stage ls (Pass<LOGN, P> of the kernels)
    const int np = (logn + CKKS_NTT_RMAX - 1) / CKKS_NTT_RMAX, base = logn / np, extra = logn % np;
    int p = 0, start = 0, len = base + (0 < extra ? 1 : 0);
    while (ls >= start + len) {
        start += len;
        ++p;
        len = base + (p < extra ? 1 : 0);
    }
    const int ep = ls - start, g = i >> ep, j = i & ((1 << ep) - 1);
    const int n_sub = cols ? 1 : 1 << log_n1;
    return (n_sub << start) + ((b * ((1 << len) - 1) + (1 << ep) - 1 + j) << start) + g;
}

static int phase_geometry(const Context &C, bool cols, NttPhase &P, PhaseLaunch &G) {
    int log_n1, log_n2;
    ntt_geometry(C.log_n, log_n1, log_n2);
    P.N = C.N;
    P.N1 = 1 << log_n1;
    P.N2 = 1 << log_n2;
    P.log_n2 = log_n2;
    P.mods = C.d_mods;
    P.tw_fwd = C.d_tw_fwd;
    P.tw_inv = C.d_tw_inv;
    G.s = phase_shape(C.log_n, cols, C.tune_ntt_tile_cols, C.tune_ntt_tile_blocks);
    return G.s.logn;
}

// One phase. phase 0 = the first phase executed (forward: columns; inverse:
// blocks), phase 1 = the second. With log_n1 == 0 there is only phase 1 work
// done as a single block phase over the whole limb.
cudaError_t launch_ntt_phase(const Context &C, bool fwd, bool cols, const LimbJobs &J, const LoadSpec &L,
                             const StoreSpec &S, cudaStream_t st) {
    NttPhase P;
    PhaseLaunch G;
    const int logn = phase_geometry(C, cols, P, G);
    G.st = st;
    count_op(C, fwd ? OP_NTT_PHASE : OP_INTT_PHASE);
    count_kernel(C);
    // algorithmic bytes: every launch limb read and written once, plus the
    // extra limbs its fused load / store touch
    const double limb = (double)C.N * sizeof(u64);
    const double jobs_d = (double)J.n_batch * J.n_polys * J.n_limbs;
    const double bp = (double)J.n_batch * J.n_polys;
    double bytes = 2.0 * jobs_d * limb;
    if (L.mode == LD_ADD) bytes += jobs_d * limb;
    if (L.mode == LD_EQ17) bytes += bp * L.mu * limb;
    if (L.mode == LD_BCONVK) bytes += bp * L.K * limb - jobs_d * limb;
    if (S.mode == ST_MODDOWN) bytes += bp * S.K * limb;
    if (S.mode == ST_MRS) bytes += jobs_d * limb;
    if (S.mode == ST_ADDSUB) bytes += 2.0 * jobs_d * limb;
    // integer work: one Shoup product per butterfly (log2 n stages of N / 2
    // per limb) plus the Shoup products of the fused load / store
    double ops = jobs_d * (double)C.N * 0.5 * logn;
    if (L.mode == LD_SIGNED) ops += jobs_d * (double)C.N;
    if (L.mode == LD_EQ17) ops += jobs_d * (double)C.N * (L.mu + L.with_self);
    if (S.mode == ST_SCALE || S.mode == ST_MODDOWN || S.mode == ST_MRS) ops += jobs_d * (double)C.N;
    ProfScope ps(C, fwd ? (cols ? KC_NTT_FWD_COLS : KC_NTT_FWD_BLOCKS) : (cols ? KC_NTT_INV_COLS : KC_NTT_INV_BLOCKS),
                 bytes, st, ops);
    if (P.N1 == 1)
        return fwd ? ntt_whole_uf(logn, P, &J, nullptr, 0, L, S, G) : ntt_whole_ui(logn, P, &J, nullptr, 0, L, S, G);
    if (C.q1() && C.log_n >= 14)
        return fwd ? ntt_two_uf1(logn, P, &J, nullptr, 0, L, S, G) : ntt_two_ui1(logn, P, &J, nullptr, 0, L, S, G);
    return fwd ? ntt_two_uf(logn, P, &J, nullptr, 0, L, S, G) : ntt_two_ui(logn, P, &J, nullptr, 0, L, S, G);
}

// One phase over a device table of limbs (cross-shape launches). The caller
// counts the algorithmic bytes and Shoup products (they depend on the
// table's entries).
cudaError_t launch_ntt_phase_table(const Context &C, bool fwd, bool cols, const NttJob *jobs, int n_jobs,
                                   const LoadSpec &L, const StoreSpec &S, double alg_bytes, double ops,
                                   cudaStream_t st) {
    if (n_jobs <= 0) return cudaSuccess;
    NttPhase P;
    PhaseLaunch G;
    const int logn = phase_geometry(C, cols, P, G);
    G.st = st;
    count_op(C, fwd ? OP_NTT_PHASE : OP_INTT_PHASE);
    count_kernel(C);
    ProfScope ps(C, fwd ? (cols ? KC_NTT_FWD_COLS : KC_NTT_FWD_BLOCKS) : (cols ? KC_NTT_INV_COLS : KC_NTT_INV_BLOCKS),
                 alg_bytes, st, ops);
    if (P.N1 == 1)
        return fwd ? ntt_whole_tf(logn, P, nullptr, jobs, n_jobs, L, S, G)
                   : ntt_whole_ti(logn, P, nullptr, jobs, n_jobs, L, S, G);
    if (C.q1() && C.log_n >= 14)
        return fwd ? ntt_two_tf1(logn, P, nullptr, jobs, n_jobs, L, S, G)
                   : ntt_two_ti1(logn, P, nullptr, jobs, n_jobs, L, S, G);
    return fwd ? ntt_two_tf(logn, P, nullptr, jobs, n_jobs, L, S, G) : ntt_two_ti(logn, P, nullptr, jobs, n_jobs, L, S, G);
}

// Full transform src -> dst with fused first load / last store. The first
// phase writes its lazy intermediate into dst (in place for the second).
cudaError_t ntt_transform(const Context &C, bool fwd, const LimbJobs &J, const LoadSpec &L, const StoreSpec &S,
                          const StoreSpec *mid, cudaStream_t st) {
    int log_n1, log_n2;
    ntt_geometry(C.log_n, log_n1, log_n2);
    count_op(C, fwd ? OP_LIMB_NTT : OP_LIMB_INTT, (unsigned long long)J.n_batch * J.n_polys * J.n_limbs);
    if (log_n1 == 0) return launch_ntt_phase(C, fwd, false, J, L, S, st);
    // first phase: forward -> columns, inverse -> blocks
    StoreSpec s1;
    if (mid) s1 = *mid;
    else { s1 = StoreSpec{}; s1.mode = ST_LAZY; s1.dst = S.dst; }
    cudaError_t e = launch_ntt_phase(C, fwd, fwd, J, L, s1, st);
    if (e != cudaSuccess) return e;
    // second phase reads the intermediate from s1.dst at the destination slots
    LimbJobs J2 = J;
    for (int i = 0; i < J.n_limbs; ++i) J2.slot[i] = J.dslot[i];
    LoadSpec l2{};
    l2.mode = LD_PLAIN;
    l2.a = s1.dst;
    return launch_ntt_phase(C, fwd, !fwd, J2, l2, S, st);
}

}  // namespace ckks
