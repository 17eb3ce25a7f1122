// The line of output tiles that wgrad_stream_kernel cuts into equal pieces, and the addition of the partial tiles.
#pragma once
#include "common.cuh"
#include "wgrad_line.h"

namespace uoe {

// One family of weight-gradient matrices [M, N], one per expert.
struct WProblem {
    int M, N, BN, m_tiles, n_tiles;
    int w;                    // cost of one 64-row K block of a tile (wgrad_tile_shape)
    int transposed;           // out[0] is [n, N, M]
    int out_cols;             // columns per output tensor (N, or N / 3 with three tensors side by side)
    float* out[3];            // [n, M, out_cols]
};
// What a launch leaves to be added (blocks = 0: nothing).
struct WReduce {
    WProblem prob[2];
    const int* offsets = nullptr;
    const float* part = nullptr;
    int n = 0, nprob = 0, pieces = 0, blocks = 0;
    int per = 1;              // blocks per tile
    int part_floats = 0;      // of a part of a tile in the scratch
    int by_cut = 0;           // blocks are counted by piece boundary (more tiles than pieces), else by tile
    int threads = 512;        // of a block
    int halves = 0, places = 0;      // half pieces of the widest tile; boundaries or tiles that blocks are counted by
    // the blocks for `t` threads each, a warp per half piece
    void use_threads(int t) { threads = t; per = (halves + t / 32 - 1) / (t / 32); blocks = places * per; }
};

constexpr int kReduceThreads = 512;      // of a block, at most

#ifdef __CUDACC__
struct WSched {
    int n, total, Q;          // cost of the line, cost of a piece
    int kb[32];               // 64-row K blocks of each expert
    int base[2][33];          // where expert e's tiles of problem p begin
};
// A tile's part inside one piece.
struct WFrag {
    int p, e, m0, n0, cols;            // problem, expert, first row and column of the tile, its columns
    int kb_lo, kb_hi;                  // K blocks of this part (none: the part is zero)
    int c_first, c_last;               // pieces that hold parts of the tile
};

// One warp builds it (n <= 32).
__device__ __forceinline__ void wsched_build(WSched& s, const int* offs, int n, const WProblem* prob, int nprob, int pieces, int lane) {
    const int kb = lane < n ? (offs[lane + 1] - offs[lane]) / 64 : 0;
    const int kb1 = lane < n ? max(kb, kMinTileKb) : 0;
    int incl = kb1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    const int all = __shfl_sync(0xffffffffu, incl, 31);
    int start = 0, wmax = 1;
    for (int p = 0; p < nprob; ++p) {
        const int per = prob[p].m_tiles * prob[p].n_tiles * prob[p].w;
        if (lane < n) s.base[p][lane] = start + (incl - kb1) * per;
        start += all * per;
        if (lane == 0) s.base[p][n] = start;
        wmax = max(wmax, prob[p].w);
    }
    if (lane < n) s.kb[lane] = kb;
    if (lane == 0) {
        s.n = n;
        s.total = start;
        s.Q = max((start + pieces - 1) / pieces, kMinPieceKb * wmax);
    }
    __syncwarp();
}
// The tile of problem p, expert e, index t within the expert; its place on the line.
__device__ __forceinline__ void wsched_tile(const WSched& s, const WProblem& pr, int p, int e, int t, WFrag& f, int& begin, int& cost) {
    const int kb1 = max(s.kb[e], kMinTileKb);
    cost = kb1 * pr.w;
    begin = s.base[p][e] + t * cost;
    f.p = p; f.e = e;
    f.m0 = (t / pr.n_tiles) * 128;
    f.n0 = (t % pr.n_tiles) * pr.BN;
    f.cols = min(pr.BN, pr.N - f.n0);
    f.c_first = begin / s.Q;
    f.c_last = (begin + (kb1 - 1) * pr.w) / s.Q;
}
// Next part of piece c at or behind pos (pos is advanced past it); false at the piece's end.  K block i of a tile that
// begins at b belongs to piece (b + i w) / Q.
__device__ __forceinline__ bool wsched_next(const WSched& s, const WProblem* prob, int c, int& pos, WFrag& f) {
    const int end = min(s.total, (c + 1) * s.Q);
    while (pos < end) {
        const int p = pos >= s.base[0][s.n] ? 1 : 0;
        int e = 0;
        while (pos >= s.base[p][e + 1]) ++e;
        const WProblem& pr = prob[p];
        const int cost1 = max(s.kb[e], kMinTileKb) * pr.w;
        int begin, cost;
        wsched_tile(s, pr, p, e, (pos - s.base[p][e]) / cost1, f, begin, cost);
        f.kb_lo = (pos - begin + pr.w - 1) / pr.w;
        f.kb_hi = min(cost / pr.w, (min(end, begin + cost) - begin + pr.w - 1) / pr.w);
        pos = begin + cost;
        if (f.kb_lo < f.kb_hi) {
            f.kb_lo = min(f.kb_lo, s.kb[e]);
            f.kb_hi = min(f.kb_hi, s.kb[e]);
            return true;
        }
    }
    return false;
}
// Scratch slot of a cut tile's part in piece c: a piece holds at most two, its first part (the tile began earlier) and its
// last (the tile goes on).
__device__ __forceinline__ size_t wsched_slot(const WFrag& f, int c) { return (size_t)c * 2 + (c > f.c_first ? 0 : 1); }

// Adds the parts of every cut tile in ascending order.  r.per blocks of r.threads threads for a tile, half a [32 x 32]
// piece per warp.  The blocks are counted by tile or, when there are more tiles than pieces, by the boundaries between
// pieces: each cuts at most one tile, whose first boundary does the work.  Bound by the latency of the part loads: two
// parts are in flight per warp (one part and a whole piece per warp: 32 us instead of 21 for the image block's MLP half).
__device__ __forceinline__ void wgrad_reduce(const WReduce& r, int blk) {
    __shared__ WSched s;
    __shared__ int offs[34];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {
        offs[lane] = r.offsets[min(lane, r.n)];
        if (lane == 0) offs[r.n] = r.offsets[r.n];
        __syncwarp();
        wsched_build(s, offs, r.n, r.prob, r.nprob, r.pieces, lane);
    }
    __syncthreads();
    WFrag f;
    int p = 0, begin, cost;
    if (r.by_cut) {
        const int c = 1 + blk / r.per, pos = c * s.Q;
        if (pos >= s.total) return;
        p = pos >= s.base[0][s.n] ? 1 : 0;
        int e = 0;
        while (pos >= s.base[p][e + 1]) ++e;
        wsched_tile(s, r.prob[p], p, e, (pos - s.base[p][e]) / (max(s.kb[e], kMinTileKb) * r.prob[p].w), f, begin, cost);
        if (f.c_first != c - 1) return;
    } else {
        const int tiles0 = r.n * r.prob[0].m_tiles * r.prob[0].n_tiles;
        int tile = blk / r.per;
        if (tile >= tiles0) { p = 1; tile -= tiles0; }
        const int per_e = r.prob[p].m_tiles * r.prob[p].n_tiles;
        wsched_tile(s, r.prob[p], p, tile / per_e, tile % per_e, f, begin, cost);
    }
    const WProblem& pr = r.prob[p];
    const int piece = (blk % r.per) * (r.threads / 32) + warp;
    const int h = piece & 1, quarter = (piece >> 1) & 3, ch = piece >> 3;
    if (f.c_first == f.c_last || ch * 32 >= f.cols) return;
    // lanes over (row, four columns) so that both the reads and the row-major writes are whole sectors; a transposed
    // output takes lanes over rows
    const int lr = pr.transposed ? lane : lane >> 3, lq = pr.transposed ? 0 : lane & 7;
    const int stride = pr.transposed ? 128 : 4;
    const float4* base = (const float4*)r.part + (size_t)ch * 8 * 128 + quarter * 32 + (pr.transposed ? 4 * h * 128 : lq * 128 + 4 * h * 4) + lr;
    auto part = [&](int c) { return base + wsched_slot(f, c) * (size_t)(r.part_floats / 4); };
    float4 acc[4], t[4];
    {
        const float4 *s0 = part(f.c_first), *s1 = part(f.c_first + 1);
#pragma unroll
        for (int q = 0; q < 4; ++q) { acc[q] = s0[q * stride]; t[q] = s1[q * stride]; }
    }
    auto add = [&](const float4* v) {
#pragma unroll
        for (int q = 0; q < 4; ++q) { acc[q].x += v[q].x; acc[q].y += v[q].y; acc[q].z += v[q].z; acc[q].w += v[q].w; }
    };
    add(t);
    for (int c = f.c_first + 2; c <= f.c_last; c += 2) {
        const bool two = c < f.c_last;
        const float4 *s0 = part(c), *s1 = part(two ? c + 1 : c);
        float4 t1[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) { t[q] = s0[q * stride]; t1[q] = s1[q * stride]; }
        add(t);
        if (two) add(t1);
    }
    const int col = f.n0 + ch * 32;
    if (pr.transposed) {
        float* o = pr.out[0] + ((size_t)f.e * pr.N + col + 16 * h) * pr.M + f.m0 + quarter * 32 + lr;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            o[(size_t)(4 * q) * pr.M] = acc[q].x; o[(size_t)(4 * q + 1) * pr.M] = acc[q].y;
            o[(size_t)(4 * q + 2) * pr.M] = acc[q].z; o[(size_t)(4 * q + 3) * pr.M] = acc[q].w;
        }
    } else {
        const int which = col / pr.out_cols;
        float* o = pr.out[which] + ((size_t)f.e * pr.M + f.m0 + quarter * 32) * pr.out_cols + (col - which * pr.out_cols) + lq * 4;
#pragma unroll
        for (int q = 0; q < 4; ++q) *(float4*)(o + (size_t)((4 * h + q) * 4 + lr) * pr.out_cols) = acc[q];
    }
}
#endif

}  // namespace uoe
