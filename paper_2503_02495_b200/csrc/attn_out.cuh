// Write-out of the expert output z by the warps of the attention kernels.
#pragma once
#include "tc.cuh"

namespace uoe {
namespace tc {

// One warp's [32 rows x 64 columns] piece of z, row `lane` in this thread: bf16 into the warp's 4 KB of staging (128-byte rows,
// swizzled), then one tensor store; with fewer than 32 rows left in the pair (the next pair's follow), eight lanes per row
// write the valid ones.  (Every piece back out of shared memory with 16-byte stores: image block forward 208.0 us, so 205.7.)
__device__ __forceinline__ void store_z_piece(const float* zf, uint8_t* stg, const CUtensorMap* tmZ, __nv_bfloat16* z, int d, int col, int row,
                                              int rows_left, int lane) {
    uint4 w[8];
#pragma unroll
    for (int ch = 0; ch < 8; ++ch) {
        w[ch].x = pack_bf16x2(zf[ch * 8 + 0], zf[ch * 8 + 1]); w[ch].y = pack_bf16x2(zf[ch * 8 + 2], zf[ch * 8 + 3]);
        w[ch].z = pack_bf16x2(zf[ch * 8 + 4], zf[ch * 8 + 5]); w[ch].w = pack_bf16x2(zf[ch * 8 + 6], zf[ch * 8 + 7]);
    }
    if (lane == 0) bulk_wait_read();                         // the previous piece has been read
    __syncwarp();
#pragma unroll
    for (int ch = 0; ch < 8; ++ch) *(uint4*)(stg + lane * 128 + ((ch ^ (lane & 7)) << 4)) = w[ch];
    if (rows_left >= 32) {                                   // (uniform over the warp)
        fence_async_smem();
        __syncwarp();
        if (lane == 0) { tma_store_2d(tmZ, stg, col, row); bulk_commit(); }
    } else {
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = i * 4 + (lane >> 3), ch = lane & 7;
            if (r < rows_left) *(uint4*)(z + (size_t)(row + r) * d + col + ch * 8) = *(const uint4*)(stg + r * 128 + ((ch ^ (r & 7)) << 4));
        }
    }
}

// The same piece straight from registers: a row's 128 bytes per thread, in whole sectors.  Where two CTAs share an SM its copy
// engine is busy with the loads of the one while the other writes z, and tensor stores queue behind them (image block forward
// 200.5 us with tensor stores, 192.3 so); with one CTA per SM tensor stores are the better ones (one sequence 55.4 against 56.4).
__device__ __forceinline__ void store_z_direct(const float* zf, __nv_bfloat16* z, int d, int col, int row, int rows_left, int lane) {
    if (lane >= rows_left) return;
    __nv_bfloat16* o = z + (size_t)(row + lane) * d + col;
    const bool whole = sector_aligned(o);
#pragma unroll
    for (int q = 0; q < 4; ++q) st_sector(o + 16 * q, pack16<__nv_bfloat16>(zf + 16 * q), pack16<__nv_bfloat16>(zf + 16 * q + 8), whole);
}

}  // namespace tc
}  // namespace uoe
