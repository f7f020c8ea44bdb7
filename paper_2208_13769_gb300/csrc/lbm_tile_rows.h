// lbm_tile_rows.h -- rows of the interior kernel's tiles: how a rectangle's
// rows are cut into chunks, and how many of them a tile may have (host code
// that needs no CUDA header).
#pragma once

#include <stdint.h>
#include <string.h>

namespace lbm {

// The rows of a rectangle as chunks: count[k] chunks of rows[k] rows for each
// level k in turn (the last of them clipped to the rectangle).
struct ChunkLevels {
    int32_t rows[4], count[4];
};

inline ChunkLevels equal_chunks(int h, int rows) {
    ChunkLevels L;
    memset(&L, 0, sizeof(L));
    L.rows[0] = rows < h ? rows : h;
    L.count[0] = (h + L.rows[0] - 1) / L.rows[0];
    return L;
}

// The most rows an interior tile may have in planes of this pitch.  The tile
// addresses its stores by 32-bit byte offsets from the node two rows and two
// columns before its first; the widest element, of `word` bytes (8 in FP64,
// else 4), that it stores lies rows + 1 pitches and fewer than `threads`
// elements above.  A plane has fewer than 2^31 elements and, if an interior
// tile exists, 14 rows or more with their padding, so that the limit is 2 or
// more (59.7e6 nodes to a row in FP64: 7).
inline int interior_max_rows(int64_t pitch, int word, int threads) {
    const int64_t elements = (int64_t(1) << 32) / word - threads;
    const int64_t rows = elements / pitch - 1;
    return rows > (1 << 20) ? 1 << 20 : int(rows);
}

// L, or equal chunks of max_rows rows where a tile of L would have more.
inline ChunkLevels bounded_chunks(const ChunkLevels& L, int h, int max_rows) {
    for (int k = 0; k < 4; ++k)
        if (L.count[k] > 0 && L.rows[k] > max_rows && h > max_rows) return equal_chunks(h, max_rows);
    return L;
}

}  // namespace lbm
