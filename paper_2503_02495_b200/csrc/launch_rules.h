// Rules by which launches choose between kernels, as far as they are arithmetic on sizes (host only).
#pragma once

namespace uoe {

constexpr int kRowTile = 128;      // rows of a tile of the grouped GEMMs; expert regions are multiples of it

// Fewest 128-row tiles that the regions of n experts can have, from the host's bound on their rows: R routed rows and at most 127 rows
// of padding per expert, in whole tiles.
inline long long least_row_tiles(long long rows_max, int n) {
    const long long t = rows_max / kRowTile - n + 1;
    return t > 0 ? t : 0;
}

// Projections to q, k and v of 128 columns each: one 384-column tile per row tile (true) or three 128-column tiles.  The
// three are the better ones while they are one wave over the SMs (block forward, 48 row tiles, d = 1024: 93.1 us, as one tile 95.2; d = 512
// 68.9 and 71.6), the one from there on (52 row tiles: 99.4 and 91.5; 128: 148.3 and 134.3).
inline bool qkv_as_one_tile(long long rows_max, int n, int sms) { return 3 * least_row_tiles(rows_max, n) > sms; }

}  // namespace uoe
