// Launch shapes of the NTT's phases: a ring degree and the tile tunables give
// CTAs, threads and shared memory. Plain C++, also compiled by the host tests.
#pragma once
#include <algorithm>
#include <cstddef>

namespace ckks {

// COLS: the column phase, BLOCKS: the block phase (and N <= 2^8 as one block),
// WHOLE: all stages of a limb in one CTA (ntt_kernel.cuh).
enum Shape { COLS = 0, BLOCKS = 1, WHOLE = 2 };
constexpr int kWholeMax = 12;  // log2 of the largest limb one CTA transforms

// Threads per CTA the kernels are compiled for.
constexpr int kPhaseThreads = 256;

// Elements per CTA of the block phases unless tuned otherwise. Their warps do
// not wait for each other, so a CTA is only the unit in which shared memory is
// given out: small CTAs start as soon as their few warps' memory is free
// (forward / inverse block phase of 384 limbs at N = 2^16: 133 / 126 us with 512
// or 1024 elements, 133 / 127 with 2048, 154 / 144 with 4096).
constexpr int kBlockTile = 1024;

// Limbs per CTA of the transforms of N <= 2^8, one per warp (2048 limbs of
// 2^7 / 2^8 points forward: 8.6 / 9.7 us with four, 10.1 / 11.6 with one, of
// which some 8 us are the call's own; with run-time modes and shared memory for
// as many blocks as a warp could hold, 10.1 / 12.3).
constexpr int kTinyLimbs = 4;

// Geometry of the phases for a given log N: log_n1 = 0 (one phase) up to
// N = 2^12, the largest limb one CTA holds.
inline void ntt_geometry(int logN, int &log_n1, int &log_n2) {
    if (logN <= kWholeMax) { log_n1 = 0; log_n2 = logN; }
    else { log_n1 = logN / 2; log_n2 = logN - log_n1; }
}

struct PhaseShape {
    int shape, logn;     // log2 of the sub-transforms' points
    int tiles, threads;  // CTAs per limb, threads per CTA
    int limbs;           // limbs per CTA
    size_t smem;
};

// One phase of the transform of N = 2^logN. A thread takes 16 points; the tile
// tunables set the elements per CTA: whole groups of 16 columns, whole warps of
// blocks, at most kPhaseThreads threads.
inline PhaseShape phase_shape(int logN, bool cols, int tile_cols, int tile_blocks) {
    int log_n1, log_n2;
    ntt_geometry(logN, log_n1, log_n2);
    const int N1 = 1 << log_n1, N2 = 1 << log_n2;
    PhaseShape S;
    S.logn = cols ? log_n1 : log_n2;
    S.limbs = 1;
    const int n = 1 << S.logn;
    const int sets = n >= 16 ? n / 16 : 1;                      // threads per sub-problem
    const size_t data = (n + n / 16) * 8, twiddles = (n - 1) * 16;  // of one block (one pad word per 16)
    S.shape = cols ? COLS : S.logn > 8 ? WHOLE : BLOCKS;
    if (S.shape == COLS) {
        const int group = 16 * sets;
        const int groups = std::max(1, std::min(tile_cols / (16 * n), std::min(kPhaseThreads / group, N2 / 16)));
        S.tiles = N2 / 16 / groups;
        S.threads = groups * group;
        S.smem = (size_t)groups * 16 * n * 8 + (size_t)n * 16;
    } else if (S.shape == WHOLE) {
        S.tiles = 1;
        S.threads = sets;
        S.smem = data + twiddles;
    } else if (log_n1 == 0) {
        S.tiles = 1;
        S.limbs = kTinyLimbs;
        S.threads = 32 * kTinyLimbs;
        S.smem = kTinyLimbs * ((data + 15) / 16 * 16 + twiddles);
    } else {
        const int threads = std::max(32, std::min(std::min(tile_blocks / 16, kPhaseThreads), N1 * sets));
        const int blocks = threads / sets;
        S.tiles = (N1 + blocks - 1) / blocks;
        S.threads = threads;
        S.smem = blocks * (data + twiddles);  // Geo::warp_bytes per warp
    }
    return S;
}

}  // namespace ckks
