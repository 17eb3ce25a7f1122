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

// Threads of the launch that turns gate gradients into the router's logit gradient (a CTA per sample, whose warps share its k c slabs)
// and adds up the cut weight-gradient tiles in further CTAs.  512 where those are many (by_cut: every block builds the line again; wide
// block, training step 504 us, with 256 threads and twice the blocks 507) and where a sample's slabs are a long chain; else
// 256, so that all CTAs are resident at once (language-model block 250.8 -> 248.2, image block 671 -> 670).  A chain is long from 224 slabs
// on where the samples are few, later where there are many of them to be resident.  Training steps of the MLP half, d = 512, 256 / 512
// threads, us: 8 samples of 200 slabs 138.2 / 138.4, of 240 145.6 / 141.6, 2 of 224 92.4 / 89.7, 16 of 360 228.3 / 220.7, 4 of 1280 314 / 286; 24 of 200
// slabs 309 / 313, of 240 332 / 336, of 256 362 / 366, 40 of 280 354.3 / 356.0, 64 of 320 489.1 / 487.3, 100 of 320 712 / 711.
inline int router_grad_threads(bool by_cut, int samples, long long slabs) {
    return by_cut || slabs >= (samples <= 16 ? 224 : 320) ? 512 : 256;
}

}  // namespace uoe
