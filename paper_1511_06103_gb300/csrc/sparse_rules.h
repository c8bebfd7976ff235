// sparse_rules.h -- how the edge-list step (sparse.cu) deals variables and
// adjacency lists out to lanes, warps and blocks.  Plain C++ (no CUDA headers), so
// that the arithmetic is checked on the CPU at sizes no test allocates:
// crf_create takes up to 2^31 - 1 variables, so index arithmetic past N is
// unsigned (a stride is below 2^18) and sums that may pass 2^31 are 64-bit.
#pragma once

#include <algorithm>
#include <cstdint>

#ifdef __CUDACC__
#define PROXMF_HD __host__ __device__
#else
#define PROXMF_HD
#endif

namespace proxmf {

constexpr int kSparseWarps = 8;                // warps per block
// Blocks per instance at most: those that run at a time on the 152 SMs, by the
// kernel's registers.  (In a batch every instance has that many, so that its free
// energy has the same bits as alone; they run in whole waves.)  With four an SM for
// asymmetric mu too, a third of whose blocks then ran in a second wave, 20 steps on
// N = 262144 with 8 entries a list took 3100 us at 21 labels, now 2230, and 612 at 8, now 515.
PROXMF_HD constexpr int sparse_per_sm(bool sym) { return sym ? 4 : 3; }
constexpr int sparse_resident(bool sym) { return 152 * sparse_per_sm(sym); }

// Lanes that hold the labels of one variable (LP stored labels, a vector each).
PROXMF_HD constexpr int sparse_lanes(int LP) { return LP <= 4 ? 1 : LP <= 8 ? 2 : LP <= 16 ? 4 : 8; }

// Lane groups per adjacency list: as many as it takes to have about 98304
// threads (20 warps per SM), but no more than half the mean list length, so
// that a group has at least two entries of its own on average.  `entries` are
// those of the longer of the two adjacency arrays.
inline int sparse_split(int N, int lanes, int64_t entries) {
    int split = 1;
    while (2 * split * lanes <= 32 && (int64_t)N * lanes * split < 98304 && entries >= (int64_t)4 * split * N)
        split *= 2;
    return split;
}

// A warp takes as long as its longest list, and a list's groups take four entries
// each in turn.  Lists longer than sparse_long_list are walked by a warp of their
// own: eight turns of its groups, and four times the mean (below that the warps are
// evenly loaded).  Lists longer than sparse_block_list are walked by a block: 16 turns
// of a warp.  Neither is done unless the longest takes 24 turns of its groups: the
// passes over the variables that it takes cost the other lists 5 to 8 %.
// us for 10 steps, with these passes / without: N = 131072 and one list of 1e5, L = 2
// 630 / 70000, L = 21 4940 / 104000; N = 262144, lists by a power law (rank ^ -0.8),
// L = 2 312 / 13200, L = 21 2230 / 24500; three lists of 100 among lists of 8, L = 2
// 183 / 217, L = 21 841 / 847, but three of 60 at L = 21 834 / 800.  16 turns in place
// of eight: 342 for the power law at L = 2; four turns: 14 % lost on random graphs
// whose longest lists are four times the mean.
inline int sparse_block_list(int lanes) { return 2048 / lanes; }
inline int sparse_long_list(int N, int lanes, int split, int64_t entries, int longest) {
    const int64_t own = lanes * split >= 32 ? sparse_block_list(lanes)   // every list has a warp
                                            : std::max<int64_t>(32 * split, 4 * entries / N);
    return longest > 3 * own ? (int)own : INT32_MAX;
}

// Blocks, and free-energy partials, per instance.
inline int sparse_blocks(int N, int lanes, int split, bool sym) {
    const int64_t per = kSparseWarps * 32 / (lanes * split);
    return (int)std::min<int64_t>((N + per - 1) / per, sparse_resident(sym));
}
inline int sparse_max_blocks(int N) {
    return (int)std::min<int64_t>(((int64_t)N + kSparseWarps - 1) / kSparseWarps, sparse_resident(true));
}

// The items a warp takes: first, first + stride, ... below n, `per` at a time.
struct SparseWalk {
    uint32_t first, stride;
};
PROXMF_HD inline SparseWalk sparse_walk(uint32_t block, uint32_t blocks, uint32_t warp, uint32_t per) {
    return {(block * kSparseWarps + warp) * per, blocks * kSparseWarps * per};
}

// The adjacency arrays are indexed by int: n_edges edges make as many entries, or
// twice as many when a list holds both directions (symmetric mu).
inline bool sparse_entries_fit(int64_t n_edges, bool both) { return n_edges * (both ? 2 : 1) <= INT32_MAX; }

}  // namespace proxmf
