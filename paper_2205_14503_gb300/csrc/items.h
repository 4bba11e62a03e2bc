// Work items of the dense frontiers and the scans: consecutive vertex ranges.
// Host code only, apart from the CUDA headers.
#pragma once
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <thread>
#include <vector>

namespace stn {

// Degree at or above which a vertex's adjacency is processed in chunks of
// CHUNK arcs (one warp per chunk) instead of inside a 32-vertex batch.
constexpr uint32_t HEAVY_DEG = 256;
constexpr uint32_t CHUNK = 512;
// Largest vertex range of a dense work item: whatever its alignment it
// touches at most 32 bitmap words, one per lane.
constexpr uint32_t ITEM_SPAN = 992;
// Arcs per dense work item where rows are uneven: some sixteen items per warp
// of the grid, within these bounds (below one relax_group a smaller item saves
// nothing; above the upper one the slowest item shows).  R-MAT 22, weights to
// 10^5, k = 64, when the rule was drawn: 2.76 ms; four items per warp up to
// 8192 arcs 3.30.
constexpr uint64_t ITEM_ARCS_MIN = 128, ITEM_ARCS_MAX = 4096;
// A sparse bitmap's items may hold this many times the arcs (few are set).
constexpr uint64_t SPARSE_ITEM_FACTOR = 8;
// Where rows are even, nothing is gained by many items, and each costs a warp
// about 2 us of dependent loads however few bits it finds: four per warp of
// the two-block grid, and one for a sparse bitmap.  Uniform random graphs,
// sixteen items per warp against four: 400,000 vertices of degree 20, k = 37
// 1.19 -> 0.72 ms, 3 * 10^6 3.3 -> 2.9; 1.5 * 10^6 of degree 6 at a quarter of
// the default band 1.61 -> 1.07.
constexpr uint64_t EVEN_ITEMS = 4;

// Arcs per row, rounded, at least one.
inline uint64_t mean_row(uint64_t m, uint32_t n) { return std::max<uint64_t>((m + n / 2) / n, 1); }
// Rows of about the same length: cut by vertices alone.
inline bool even_rows(uint32_t max_deg, uint64_t m, uint32_t n) { return max_deg <= 4 * mean_row(m, n) + 32; }

// Cuts the vertices into consecutive ranges of about equal arcs (a hub counts
// HEAVY_DEG: longer rows are queued in chunks) and at most ITEM_SPAN vertices,
// and into coarser ones for sparse bitmaps, for a grid of `warps` warps (three
// blocks per SM); a single vertex may exceed the arc limit.  at[0] / at[1]
// receive the range starts followed by n, at[2] those of the scans, which run
// eight blocks per SM and take the finer ranges everywhere (empty: at[0]; grid
// 4096 x 4096, scan 0.355 ms in the ranges of the frontiers, 0.335).  Even rows are cut into ranges of
// equal length; else blocks of CUT_BLOCK vertices are cut side by side on the
// host's threads.  False: out of memory (nothing is thrown, on any thread).
inline bool cut_items(const uint32_t *row_ptr, uint32_t n, uint32_t max_deg, uint64_t warps,
                      std::vector<uint32_t> (&at)[3]) noexcept try {
    constexpr uint32_t CUT_BLOCK = 1u << 17;
    const uint64_t m = row_ptr[n], mean = mean_row(m, n);
    const uint64_t arcs = std::min(std::max(m / (16 * warps), ITEM_ARCS_MIN), ITEM_ARCS_MAX);
    if (even_rows(max_deg, m, n)) {
        const uint64_t two = std::max<uint64_t>(warps * 2 / 3, 1);     // warps of the two-block form
        const uint64_t span[3] = {std::max(arcs / mean, std::min(ITEM_ARCS_MAX / mean, n / (EVEN_ITEMS * two) + 1)),
                                  std::max(SPARSE_ITEM_FACTOR * arcs / mean, n / two + 1), arcs / mean};
        for (int i = 0; i < 3; ++i) {
            const uint32_t step = (uint32_t)std::min<uint64_t>(std::max<uint64_t>(span[i], 1), ITEM_SPAN);
            at[i].reserve(n / step + 2);
            for (uint64_t v = 0; v < n; v += step) at[i].push_back((uint32_t)v);
            at[i].push_back(n);
        }
        return true;
    }
    struct Part {
        std::vector<uint32_t> at[2];
    };
    const uint32_t blocks = (uint32_t)(((uint64_t)n + CUT_BLOCK - 1) / CUT_BLOCK);
    std::vector<Part> part(blocks);
    std::atomic<uint32_t> next{0};
    std::atomic<bool> failed{false};
    auto work = [&]() noexcept {
        try {
            for (uint32_t b; (b = next.fetch_add(1)) < blocks;) {
                const uint32_t lo = b * CUT_BLOCK, hi = (uint32_t)std::min<uint64_t>(n, (uint64_t)lo + CUT_BLOCK);
                const uint64_t limit[2] = {arcs, SPARSE_ITEM_FACTOR * arcs};
                uint64_t sum[2] = {0, 0};
                uint32_t from[2] = {lo, lo};
                for (int i = 0; i < 2; ++i) part[b].at[i].push_back(lo);
                for (uint32_t v = lo; v < hi; ++v) {
                    const uint32_t d = std::min(row_ptr[v + 1] - row_ptr[v], HEAVY_DEG);
                    for (int i = 0; i < 2; ++i) {
                        if (v > from[i] && (sum[i] + d > limit[i] || v - from[i] == ITEM_SPAN)) {
                            part[b].at[i].push_back(from[i] = v);
                            sum[i] = 0;
                        }
                        sum[i] += d;
                    }
                }
            }
        } catch (...) {
            failed = true;
        }
    };
    std::vector<std::thread> pool;
    const uint32_t threads = std::min(blocks, std::min(16u, std::max(1u, std::thread::hardware_concurrency())));
    try {
        pool.reserve(threads);
        for (uint32_t t = 1; t < threads; ++t) pool.emplace_back(work);
    } catch (...) {
        // fewer threads do the same work
    }
    work();
    for (auto &t : pool) t.join();
    if (failed) return false;
    for (int i = 0; i < 2; ++i) {
        size_t total = 1;
        for (auto &p : part) total += p.at[i].size();
        at[i].reserve(total);
        for (auto &p : part) at[i].insert(at[i].end(), p.at[i].begin(), p.at[i].end());
        at[i].push_back(n);
    }
    return true;
} catch (...) {
    return false;
}

}  // namespace stn
