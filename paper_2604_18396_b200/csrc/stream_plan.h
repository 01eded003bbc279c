// Launch rules of the CUDA-core streaming kernels.  Host arithmetic on sizes only, without CUDA types, so that they can be checked
// where there is no GPU.
#pragma once
#include <algorithm>

namespace river {

// 128-bit pieces of a row that a thread keeps in registers while a one-row step stages it, by weight rows per task.
template <int R> constexpr int kStreamPieces = R == 2 ? 4 : 2;
// Warps that hold a row of K inputs so.
inline int stream_hold_warps(int K, int R) {
    const int per_warp = 128 * (R == 2 ? kStreamPieces<2> : kStreamPieces<4>);
    return (K + per_warp - 1) / per_warp;
}

// Steps of up to four rows, where an SM's share of a projection is a task (R weight rows) for each of sixteen warps at most: as many warps as tasks - at least
// four, and as many as hold one row in registers - and no CTA without a task.  The other warps, of sixteen, would have nothing to
// stream, but stage the row and wait for each other with the rest, and keep the registers from whatever runs beside this grid.
// Three contexts in flight, us a step, sixteen warps everywhere against this: tiny shape, one row 61 / 40; mini 133 / 67; 1B-class,
// 4 blocks, three rows 280 / 238; one context by itself 2-10 % less or the same.  Not for lists of
// more rows, passes of four each: every pass stages its rows anew, for which all warps count (exit layers in groups of 32, mini shape,
// 64 rows: 1881 us a step so, 1704 with all of them; 1B-class, 4 blocks 1952 / 1845).
constexpr int kStreamFewRows = 4;
struct StreamGeom { int threads, grid; };
inline bool stream_small_share(int num_sms, int rows, int tasks, int K, int R, StreamGeom &g) {
    if (rows > kStreamFewRows) return false;
    const int share = (tasks + num_sms - 1) / num_sms, hold = stream_hold_warps(K, R);
    if (share > 16 || hold > 16) return false;
    g = StreamGeom{32 * std::max(std::max(4, hold), share), std::min(tasks, num_sms)};
    return true;
}

}  // namespace river
