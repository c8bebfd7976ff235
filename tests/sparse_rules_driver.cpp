// The edge-list step's walk over its variables and its launch sizes, up to the
// largest graph that a handle takes; built with UBSan.
#include <cstdio>

#include "sparse_rules.h"

using namespace proxmf;

static long bad = 0;
static void check(bool ok, const char *what, long long a, long long b) {
    if (!ok && ++bad <= 20) std::printf("%s: %lld %lld\n", what, a, b);
}

int main() {
    const int sizes[] = {1, 7, 8, 9, 255, 256, 257, 20011, 262144, 1000000, (1 << 30) + 5, 2147483647 - 155648,
                         2147483647 - 155647, 2147483647 - 256, 2147483647 - 254, 2147483647 - 7, 2147483647};
    for (int N : sizes)
        for (int lanes = 1; lanes <= 8; lanes *= 2)
            for (long long deg : {0LL, 1LL, 40LL, 3000LL}) {
                const int split = sparse_split(N, lanes, deg * N), per = 32 / (lanes * split);
                for (bool sym : {false, true}) {
                    // registers for three blocks of an SM (four with symmetric mu): no last wave that is nearly empty
                    const int resident = 152 * (sym ? 4 : 3), blocks = sparse_blocks(N, lanes, split, sym);
                    const int block = sparse_block_list(lanes), longest = N / 2;
                    const int lng = sparse_long_list(N, lanes, split, deg * N, longest);
                    check(lng == INT32_MAX || (lng >= 4 * deg && lng >= 32 && longest > lng) || lng == block, "long list", N, lng);
                    check(split >= 1 && per >= 1, "split", N, split);
                    check(blocks >= 1 && blocks <= sparse_max_blocks(N) && blocks <= resident, "blocks", N, blocks);
                    check((long long)blocks * kSparseWarps * per >= N || blocks == resident, "blocks cover N", N, blocks);
                    // the last positions of every warp: each step past them ends its loop
                    for (int b = 0; b < blocks; ++b)
                        for (int w = 0; w < kSparseWarps; ++w) {
                            const SparseWalk k = sparse_walk(b, blocks, w, per);
                            check(k.stride < (1u << 18), "stride", N, k.stride);
                            if (k.first >= (uint32_t)N) continue;
                            const long long rounds = ((long long)N - 1 - k.first) / k.stride;
                            const uint32_t last = k.first + (uint32_t)rounds * k.stride;
                            check(last < (uint32_t)N && (long long)last == k.first + rounds * k.stride, "last", N, last);
                            for (int slot = 0; slot < per; ++slot)
                                check(last + slot + k.stride >= (uint32_t)N, "past the last", N, slot);
                            check(last + k.stride >= (uint32_t)N, "loop ends", N, last);
                        }
                }
            }
    check(sparse_entries_fit(1 << 30, false) && !sparse_entries_fit(1 << 30, true) &&
              sparse_entries_fit((1 << 30) - 1, true),
          "entries", 0, 0);
    if (bad) std::printf("%ld checks failed\n", bad);
    return bad ? 1 : 0;
}
