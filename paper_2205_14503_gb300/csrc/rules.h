// Rules of dispatch that weigh measured costs, apart from the CUDA headers.
#pragma once
#include <cstdint>

namespace stn {

// Whether the tree-only scan of a graph with m arcs, weights to max_w and rows
// split at delta pays for k seeds (where it is exact).  It spares the heavy
// part of most rows, and costs a second compaction of the pair table and a
// second MST.  Query times, full against tree-only scan, in ms:
//  * below 2^27 arcs it gains little: R-MAT 22, k = 300 2.33 against 2.23,
//    R-MAT 20, k = 1000 1.42 against 1.42;
//  * fewer than three spared arcs per table entry (of uniform weights, taken
//    as 1 - 1.5 delta / max_w of the arcs: the light part is read at random):
//    k = 10,000, 1.55 * 10^8 arcs, delta at 1/2, 1/4, 1/8 and 1/32 of max_w
//    4.24 against 5.08, 3.21 against 3.68, 2.87 against 3.05, 3.27 against
//    3.10; with 5.2 * 10^8 arcs 9.16 against 9.47, 6.64 against 6.07, 5.72
//    against 4.70; k = 2000 never costs more than 6 %;
//  * bands of one to three weights hold next to no bridge, so that the rest
//    scan reads most rows: 4.30 against 5.26 (delta 2, weights to 20), 24.3
//    against 26.4 (delta 3, weights to 60); at delta 5 4.42 against 3.00.
// Elsewhere 1.0 to 1.5 times as fast: R-MAT 26 (degree 8), k = 10,000 11.0
// against 7.6, R-MAT 24, k = 700 at the default band 6.35 against 5.58.  Tables
// beyond 16,384 seeds are reached by weights to 511 alone (narrow labels).
constexpr uint64_t TREE_SCAN_MIN_ARCS = 1ull << 27;
inline bool tree_scan_pays(uint64_t m, uint32_t k, uint32_t delta, uint32_t max_w) {
    if (m < TREE_SCAN_MIN_ARCS || delta < 4) return false;
    const double slots = 0.5 * k * (k - 1.0);
    return (double)m * (1.0 - 1.5 * delta / max_w) >= 3.0 * slots;
}

// The first band's inner threshold with the split on for band width delta (0:
// none), delta0 being the default.  The default band width is 32 mean weights
// over the mean degree: on R-MAT graphs the hubs and most of the core settle
// below half a mean weight over the mean degree, and with them settled the rest
// of the band improves most vertices once.  R-MAT of 10^6 vertices, k = 101,
// default band: 54 -> 26 M relaxations, 1.72 -> 1.10 ms (1.06 at a 48th, 1.35
// at a 96th of the default width); R-MAT 24, k = 700: 11.2 -> 6.6 ms.  Bands
// narrowed by tuning gain less and take an eighth of themselves: R-MAT 26
// (degree 8), k = 10,000 14.2 -> 13.4 ms, R-MAT 22, weights to 10^5, k = 64 2.35
// -> 2.04.  Without hubs (even rows) a narrowed band gains nothing, and its
// fewer listings can keep the heavy pass from its pull form: uniform random
// graphs of lognormal weights at a 16th of the default, 30,000 vertices, k =
// 1000 0.96 -> 0.46 ms in one step, 1.5 * 10^6, k = 37 1.11 -> 1.09, 3 * 10^6,
// k = 2 1.74 -> 1.70.
inline uint32_t first_step(uint32_t delta, uint32_t delta0, uint32_t max_w, bool even) {
    if (delta > max_w) return 0;
    const bool narrowed = delta <= delta0 / 8;
    if (narrowed && even) return 0;
    const uint32_t s = narrowed ? delta / 8 : delta0 / 64;
    return s < 2 ? 2 : s;
}

}  // namespace stn
