// Pieces of a row: 32-bit arc indexes reach 2^32 - 2, so an index a piece or
// a warp's step beyond a row's end may wrap.  Pieces are therefore cut by
// their offset inside the row, and loops count a piece's arcs down.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define STN_HD __host__ __device__ __forceinline__
#else
#define STN_HD inline
#endif

namespace stn {

struct RowPiece {
    uint32_t first;      // arc index
    uint32_t count;      // arcs (0: the row ends before the piece)
};

// At most `len` arcs of the row [start, end) from offset `at` inside it.
STN_HD RowPiece row_piece(uint32_t start, uint32_t end, uint32_t at, uint32_t len) {
    const uint32_t deg = end - start;
    if (at >= deg) return RowPiece{end, 0u};
    return RowPiece{start + at, deg - at < len ? deg - at : len};
}

// End of the piece of at most `len` arcs from arc s of a row on, for the part
// of the row that ends at `end` (before s: no arcs).
STN_HD uint32_t piece_end(uint32_t s, uint32_t end, uint32_t len) {
    return end > s ? s + (end - s < len ? end - s : len) : s;
}

// The piece without its first `step` arcs.
STN_HD void skip_arcs(RowPiece &p, uint32_t step) {
    p.first += step;
    p.count -= p.count < step ? p.count : step;
}

}  // namespace stn
