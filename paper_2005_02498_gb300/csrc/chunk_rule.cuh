// chunk_rule.cuh -- how the sources of an FP64 pair evaluation are split into chunks
// (host code, plain C++).
//
// Every (target tile, chunk) is a work item; the chunks' nodal force parts, 48 bytes per node
// and chunk, are summed node by node afterwards.
#pragma once

#include <stdint.h>

#include <algorithm>
#include <vector>

namespace ptadd {

// Parts beyond this are not worth their memory: chunks grow instead.  Few targets among very many
// sources ask for the most chunks: 64 targets, 2.2e6 sources would hold 54 GB in 512 chunks.
constexpr int64_t PARTS_MAX_BYTES = (int64_t)1 << 30;
constexpr int64_t PART_BYTES = 48;  // per node and chunk

// Sources per chunk for `tiles` one-warp target tiles over n_src sources, `slots` tiles
// resident at a time (16 per SM).  Up to 16 waves of them in chunks of
// at least 64 sources (about one group of sums), so that the tail costs a few
// per cent.  Where that leaves fewer than four waves the chunks shrink to 4
// sources, and below that while a wave is not full: a lone warp spends 3.3 us
// on a source, and the FP64 near pairs of a loop (5 us per 32) sit in few
// chunks.  Measured, us per launch: 42 segments 29 / 22 in chunks of 3 / 1; 512
// segments 93 / 68 / 56 / 65 in chunks of 16 / 8 / 4 / 2; 64 targets x 1280
// sources 101 / 57 / 35 in 20 / 10 / 5; 1041 x 1485 244 / 220 / 190 in 23 / 12 /
// 6; 8192 segments 6330 / 6163 / 6155 in 128 / 64 / 32.
inline int64_t chunk_len_rule(int64_t slots, int64_t tiles, int64_t n_src)
{
    tiles = std::max<int64_t>(tiles, 1);
    int64_t ch = std::min((16 * slots + tiles - 1) / tiles, n_src / 64);
    if (tiles * ch < 4 * slots) ch = std::min((4 * slots + tiles - 1) / tiles, n_src / 4);
    if (tiles * ch < slots) ch = std::min(slots / tiles, n_src);
    ch = std::max<int64_t>(ch, 1);
    return (n_src + ch - 1) / ch;
}

// The most chunks of a single network of n nodes: 512 while their parts stay below
// PARTS_MAX_BYTES (43 690 nodes), and 64 for any size.
inline int network_max_chunks(int64_t n)
{
    return (int)std::min<int64_t>(512, std::max<int64_t>(64, PARTS_MAX_BYTES / (PART_BYTES * std::max<int64_t>(n, 1))));
}

// Sources per chunk of each realisation of a batch, n[r] nodes each, `tiles` target tiles in all:
// the rule above for the mean realisation, at most `longest`.  A realisation far above the mean gets
// at most four times the mean one's chunks: each of its nodes sums all of them, and parts and work
// items would grow as n_r^2 / mean (one of 100 000 segments among a thousand of 2: 14 GB and 9.2
// million items; so 58 MB and 39 000).  Below that the chunks are equal, which a list sorted by
// cost balances best.  All chunks grow while the parts take more than PARTS_MAX_BYTES.
inline std::vector<int64_t> batch_chunk_lens(int64_t slots, int64_t tiles, const std::vector<int64_t>& n, int64_t longest)
{
    int64_t total = 0;
    for (int64_t k : n) total += k;
    const int64_t mean = std::max<int64_t>(1, total / (int64_t)n.size()), fine = chunk_len_rule(slots, tiles, mean);
    const int64_t most = 4 * ((mean + fine - 1) / fine);
    std::vector<int64_t> len(n.size());
    for (int64_t scale = 1;; scale *= 2) {
        int64_t bytes = 0;
        bool grow = false;
        for (size_t r = 0; r < n.size(); ++r) {
            len[r] = std::min(longest, scale * std::max(fine, (n[r] + most - 1) / most));
            bytes += PART_BYTES * n[r] * ((n[r] + len[r] - 1) / len[r]);
            grow = grow || (len[r] < longest && len[r] < n[r]);
        }
        if (bytes <= PARTS_MAX_BYTES || !grow) return len;
    }
}

}  // namespace ptadd
