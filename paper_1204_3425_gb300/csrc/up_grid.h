// Grid of the resident-row up phase (host code without CUDA, so that a CPU test
// can walk it over every sector).
#ifndef HUB_UP_GRID_H
#define HUB_UP_GRID_H
#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace hub {

struct UpGrid {
    int gx, gy;                      // row ranges, interleaved column chunks; gx * gy <= the CTAs asked for
    int64_t rows;                    // of a range, on average
    int cap;                         // rows whose lists fit in shared memory at a time
    int W;                           // longest hop list
    size_t smem;
};

// Cost of a row's segment in units of one hop, besides its hops.
constexpr int kUpRowCost = 8;

// Row ranges and column groups: ranges of about 32 rows, the chunks dealt to as
// many CTAs of each range as the device holds (never more in all, also where a
// sector has fewer rows than a range: with one spin empty or full it has one row).
// Longer ranges let a list serve more segments, but the CTAs then differ more in
// how their memory rounds add up (4x4 (5,5) binary64: 403, 385, 376, 392, 414 us
// with 7, 14, 29, 57, 115 rows; 4x4 (8,8) binary32: 1.95, 1.91, 1.97, 2.01 ms with
// 21, 42, 85, 169).  The chunks are dealt evenly: 15 of them to 12 groups leave
// nine CTAs in twelve idle half the time (ring 13 (6,6): binary32 product 31.8 ->
// 25.9 us with 8 groups, binary64 60.6 -> 54.4).  hops: of all rows; W: of the longest.
inline UpGrid make_up_grid(int64_t Dup, int64_t hops, int W, int64_t nchunk, int ctas) {
    UpGrid g;
    g.W = std::max(W, 1);
    g.gy = (int)std::max<int64_t>(1, std::min<int64_t>({nchunk, (int64_t)ctas, (32 * (int64_t)ctas + Dup - 1) / Dup}));
    const int64_t rounds = (nchunk + g.gy - 1) / g.gy;         // chunks of a CTA; no fewer CTAs than that takes
    g.gy = (int)((nchunk + rounds - 1) / rounds);
    g.gx = (int)std::max<int64_t>(1, std::min<int64_t>(ctas / g.gy, (Dup + 7) / 8));
    // most rows of a range: all of them without hops
    const int64_t total = hops + kUpRowCost * Dup;
    const int64_t rows = std::min<int64_t>(Dup, total / g.gx / kUpRowCost + 2);
    g.rows = (Dup + g.gx - 1) / g.gx;
    const int64_t per_row = 12 + 4 * (int64_t)g.W;
    g.cap = (int)std::max<int64_t>(1, std::min<int64_t>(rows, 24 * 1024 / per_row));
    g.smem = (size_t)(g.cap * per_row);
    return g;
}

}  // namespace hub
#endif
