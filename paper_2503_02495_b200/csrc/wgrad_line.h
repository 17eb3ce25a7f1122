// Host arithmetic of the line of output tiles that wgrad_stream_kernel cuts into pieces (plain C++, no CUDA types, so that it
// can be compiled and tested on its own).
#pragma once

namespace uoe {

// A tile counts as at least this many K blocks: writing its 128 KB out takes about as long, and an expert with few or no
// rows has as many tiles as any other (uncounted, one CTA wrote all of an empty expert's zeros: 78 us instead of 50 for
// the MLP half at B = 4, L = 2048, d = 1024, d_e = 512, n = 8 with one expert unused).
constexpr int kMinTileKb = 4;
constexpr int kLineBK = 64;          // rows of a K block
constexpr int kLineBM = 128;         // rows of an output tile
constexpr int kLineBNMax = 256;      // its columns at most
// The cost of a K block is kStepCost plus one per 64 columns of either operand: a block takes 1000 to 1500 cycles, most
// of it the round trip of its copies whatever their width.  With the bytes alone as the cost (no constant part) the
// pieces of narrow tiles were the last to end: image block, training 749 us -> 742, language-model block 279 -> 277.
constexpr int kStepCost = 16;

// Output tiles of one expert's [M, N] gradient: 128 rows, column tiles of at most 256, as equal as 64-wide blocks allow.
struct WTileShape { int m_tiles, n_tiles, BN, w /* cost of one K block of a tile */; };
inline WTileShape wgrad_tile_shape(int M, int N) {
    WTileShape t;
    t.n_tiles = (N + kLineBNMax - 1) / kLineBNMax;
    t.BN = (N / 64 + t.n_tiles - 1) / t.n_tiles * 64;
    if (t.BN < 64) t.BN = 64;        // (widths the kernel refuses: only the workspace query gets here)
    t.n_tiles = (N + t.BN - 1) / t.BN;
    t.m_tiles = M / kLineBM;
    t.w = kStepCost + (kLineBM + t.BN) / 64;
    return t;
}
// Bound on the length of the line for any load of the experts: their regions have at most rows_max rows together, and an
// expert's tiles count at most kMinTileKb K blocks more than it has.
inline long long wgrad_line_bound(const WTileShape* t, int nprob, int n, long long rows_max) {
    long long cost = 0;
    for (int p = 0; p < nprob; ++p) cost += (long long)t[p].m_tiles * t[p].n_tiles * t[p].w * (rows_max / kLineBK + (long long)kMinTileKb * n);
    return cost;
}
// Pieces (one CTA each, at most one per SM of 148) that the line can fill when every piece is at least kMinPieceKb K blocks
// of the widest tile: what is launched, and what the scratch of cut tiles is sized for.
constexpr int kMaxPieces = 148, kMinPieceKb = 4;
inline int wgrad_pieces(long long bound, int wmax, int sms) {
    const long long least = (long long)kMinPieceKb * wmax, fill = (bound + least - 1) / least;
    const int cap = sms < kMaxPieces ? sms : kMaxPieces;
    return fill < 1 ? 1 : (fill < cap ? (int)fill : cap);
}
// Floats of that scratch: two parts of a tile per piece, each as wide as the widest tile.
inline long long wgrad_part_floats(int widest) { return (long long)kLineBM * widest; }
inline long long wgrad_scratch_floats(const WTileShape* t, int nprob, int n, long long rows_max) {
    int wmax = 0, widest = 0;
    for (int p = 0; p < nprob; ++p) {
        if (t[p].w > wmax) wmax = t[p].w;
        if (t[p].BN > widest) widest = t[p].BN;
    }
    return 2 * wgrad_part_floats(widest) * wgrad_pieces(wgrad_line_bound(t, nprob, n, rows_max), wmax, kMaxPieces);
}
// Whether the line and the piece ends, multiples of a piece that is rounded up, fit the kernel's 32-bit positions.
inline bool wgrad_line_fits(long long bound, int wmax, int pieces) {
    const long long rounded = bound + pieces, least = (long long)kMinPieceKb * wmax * pieces;      // pieces * Q, Q = max(ceil(line / pieces), kMinPieceKb wmax)
    return (rounded > least ? rounded : least) + wmax < 0x7fffffffll;
}

}  // namespace uoe
