// Which kernel takes a wm_checksum_xxh64 call, and its grid.  Plain C++ (host side).
#pragma once
#include <cstdint>

namespace wm {

constexpr uint32_t kXRows = 8;                          // chunks a chain warp walks at a time, at most

struct XxhPlan {
    bool paced;               // k_xxh64_paced, otherwise k_xxh64 (rows, rows0 unused)
    uint32_t blocks;
    uint32_t rows, rows0;     // chunks a block takes, and how many of them its first chain takes
};

// The paced kernel takes up to 16 chunks per block, a block per SM at a time, at 13.2 ns a stripe; rows are
// rounded up, so some SMs may have no block (149 chunks: 75 blocks of two).  With more chunks its blocks come in
// turns.  The other one takes 36 to 38 ns a stripe with 2,400 chunks, 41 to 44 with 4,700, until it is bound by
// the memory rate (from about 7,000 chunks on), so it is ahead from three turns on.  Two turns and the other kernel:
// 3,000 chunks of 1 MiB 857 us and 1196, 3,600 of 240 KiB 210 and 294, 4,736 of 64 KiB 68 and 88, of 16 KiB 25.1
// and 26.7 (2,369 of 16 KiB: 22.9 either way).
// (Divided first: for the largest counts that 32 bits hold, a sum in front of the division wraps.  n_chunks >= 1.)
inline XxhPlan xxh64_plan(uint32_t n_chunks, uint32_t n_sm)
{
    XxhPlan p = {};
    const uint32_t turns = (n_chunks - 1u) / (2u * kXRows * n_sm) + 1u;
    p.paced = turns <= 2u;
    if (p.paced) {
        p.rows = (n_chunks - 1u) / (turns * n_sm) + 1u;
        p.rows0 = p.rows <= kXRows ? p.rows : (p.rows + 1u) / 2u;
        p.blocks = (n_chunks - 1u) / p.rows + 1u;
    } else {
        p.blocks = (n_chunks - 1u) / 8u + 1u;
    }
    return p;
}

}  // namespace wm
