// Backward of the selective multi-head attention core (derivative of Eq. 33-34 with the masks of Eq. 41 and
// Fig. 4).  For every (sample, chosen expert) pair and head, with P = softmax(q k^T / sqrt(d_h) + mask),
// o = P v and the upstream gradient do:
//   dv = P^T do,   dP = do v^T,   dS = P * (dP - delta) / sqrt(d_h)  with  delta_r = sum_c do[r,c] o[r,c],
//   dq = dS k,     dk = dS^T q.
// P is rebuilt from q, k and the saved log-sum-exp of each query row, so nothing of size l_a x l_a is stored.
//
// Every output element is accumulated by a single CTA in a fixed order (no atomics).  Three forms of one kernel:
//   kSingle   l_a <= 128 (one tile of queries, one of keys): a CTA per (head, pair) makes all three gradients, S and P once
//   kDkDv     CTA = (key tile of 128, head, pair): K_j, V_j stay in shared memory, the queries stream through in blocks of
//             64; dV_j += P^T dO_i and dK_j += dS^T Q_i accumulate in TMEM
//   kDq       CTA = (query tile of 128, head, pair): Q_i, dO_i stay, the keys stream in blocks of 64; dQ_i += dS K_j
// Per step two products into TMEM (tcgen05.mma; S and dP, transposed, lanes = keys, for kSingle and kDkDv), then two threads
// per TMEM lane form P and dS, round them to bf16 and write them to shared memory in the 128B-swizzled layout, where they
// are the A operands of the second products (K-major as written, or MN-major, i.e. transposed, for kSingle's dQ).
// Bound by the chain MMA -> exponentials -> MMA of a step; so the blocks are small enough (256 TMEM columns, less than half
// of the shared memory) for two CTAs per SM, which fill each other's gaps; kDkDv and kDq run in one launch, and with the
// causal mask the CTAs with the longest streams start first.  (128 x 128 steps with one CTA per SM, and two passes also for single tiles: 50 + 38 us for 768 pairs
// of 112 tokens, 52 + 40 us for 32 causal heads of 1024 tokens.)
// Masks as in the forward kernel: key c is kept iff c < n_valid (real keys are a prefix of the gathered order)
// and, with the causal flag, c <= query row; query rows >= l_a of a tile belong to the next pair and are dropped.
#include "kernels.cuh"
#include "tc.cuh"
#include "tmap.cuh"

namespace uoe {
namespace {

using namespace tc;

constexpr int T = 128, DH = 64, TS = 64;          // rows of a resident tile; head width; rows of a streamed block
constexpr int kThreads = 256;
constexpr int TILE_BYTES = T * DH * 2;            // 16 KB: [128 x 64] bf16
constexpr int BLK_BYTES = TS * DH * 2;            // 8 KB: [64 x 64] bf16
enum BwdMode { kSingle = 0, kDkDv = 1, kDq = 2 };

// shared memory: resident tiles, streamed blocks (two stages of a pair), P and dS tiles; 1 KB that the alignment of the base
// and the control block share (so that kSingle fits an SM twice)
template <int MODE> struct BCfg {
    static constexpr int TILES = MODE == kSingle ? 4 * TILE_BYTES + 3 * TILE_BYTES           // Q K V dO | P upper half, dS (P's lower half takes V's place)
                                                 : 2 * TILE_BYTES + 4 * BLK_BYTES + (MODE == kDkDv ? 2 : 1) * TILE_BYTES;
    static constexpr int SMEM = TILES + 1024 + (MODE == kSingle ? 0 : 2048);
};

static_assert(BCfg<kDkDv>::SMEM >= BCfg<kDq>::SMEM && 2 * (BCfg<kSingle>::SMEM + 1024) <= 228 * 1024, "two CTAs per SM");

struct BCtl {
    uint64_t bar_fix, bar_ld[2], bar_s, bar_o;
    uint32_t tmem_base;
    int abort_flag;
    int n_valid;
    int pad;
};
static_assert(sizeof(BCtl) <= 128, "control block");

struct BwdArgs {
    __nv_bfloat16 *dq, *dk, *dv;
    int ld_out;                        // elements per row of the output buffers
    const float *lse, *delta;
    const int *pair_row, *patch_idx;
    int c, l_p, Lv, l_a, heads, causal, n_tiles;
    float scale_log2, inv_sqrt_dh;
    int* status;
};

struct BwdMaps { CUtensorMap q, k, v, dout; };      // [rows, d_g] in boxes of 64 columns

template <int MODE>
__device__ __forceinline__ void attn_bwd_body(const BwdMaps& m, const BwdMaps& mb /* 64-row boxes */, const BwdArgs& a, const Rope& rope, int tile) {
    const CUtensorMap *tmS0 = MODE == kDq ? &mb.k : &mb.q, *tmS1 = MODE == kDq ? &mb.v : &mb.dout;      // streamed
    extern __shared__ uint8_t smem_raw[];
    const uint32_t misalign = smem_u32(smem_raw) & 1023, lead = misalign ? 1024 - misalign : 0;
    uint8_t* smem = smem_raw + lead;
    // the control block (and the streamed rows' statistics) behind the tiles, or in the lead where that is the larger part
    uint8_t* tail = smem + BCfg<MODE>::TILES;
    BCtl* ctl = (BCtl*)(MODE == kSingle && lead > 512 ? smem_raw + ((16 - (misalign & 15)) & 15) : tail);
    float* s_stat = (float*)(tail + 128);          // kDkDv: [2 stages][lse * log2 e | delta][64]
    volatile int* abort_flag = &ctl->abort_flag;
    int* status = a.status;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t el = elect_one();               // MMAs: issued by one lane of the converged warp 0
    const int head = blockIdx.x, pair = blockIdx.y;

    if (warp == 0) tmem_alloc(&ctl->tmem_base, 256);
    if (tid == 32) {
        mbar_init(&ctl->bar_fix, 1);
        mbar_init(&ctl->bar_ld[0], 1);
        mbar_init(&ctl->bar_ld[1], 1);
        mbar_init(&ctl->bar_s, 1);
        mbar_init(&ctl->bar_o, 1);
        ctl->abort_flag = 0;
        fence_barrier_init();
    }
    pdl_wait();
    const int row_base = a.pair_row[pair];
    if (warp == 2) {                               // real keys of this pair: the real tokens of its slots' patches
        int nv = 0;
        for (int u = lane; u < a.c; u += 32) {
            const int j = a.patch_idx[(size_t)pair * a.c + u];
            if (j >= 0) nv += max(0, min(a.l_p, a.Lv - j * a.l_p));
        }
        nv = __reduce_add_sync(0xffffffffu, nv);
        if (lane == 0) ctl->n_valid = nv;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    const int kv_end = min(ctl->n_valid, a.l_a);
    const int col_h = head * DH;
    const int quarter = warp & 3, hsel = warp >> 2;                          // TMEM lane quarter; half of the columns
    const int trow = quarter * 32 + lane;                                    // TMEM lane = row of the resident tile
    const uint32_t t_lane = tmem + ((uint32_t)(quarter * 32) << 16);
    const int sw = trow & 7;
    bool ok = true;

    // P and dS of 32 columns: s <- p, dp <- ds.  Column j of the piece is kept iff lo <= j < hi; lse2 and delta belong to the
    // queries: one pair per thread (lanes = queries) or one per column, from shared memory (lanes = keys).
    auto p_and_ds = [&](float* s, float* dp, int lo, int hi, const float* lse2, const float* delta, bool per_col) {
#pragma unroll
        for (int j4 = 0; j4 < 8; ++j4) {
            float4 l4, d4;
            if (per_col) { l4 = *(const float4*)(lse2 + 4 * j4); d4 = *(const float4*)(delta + 4 * j4); }
            else { l4 = make_float4(lse2[0], lse2[0], lse2[0], lse2[0]); d4 = make_float4(delta[0], delta[0], delta[0], delta[0]); }
            const float l[4] = {l4.x, l4.y, l4.z, l4.w}, dl[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int j = 4 * j4 + q;
                const bool keep = j >= lo && j < hi;
                const float p = keep ? ex2_approx(fmaf(s[j], a.scale_log2, -l[q])) : 0.f;
                s[j] = p;
                dp[j] = keep ? p * (dp[j] - dl[q]) * a.inv_sqrt_dh : 0.f;
            }
        }
    };
    // 32 columns of this thread's row as bf16 into a swizzled [128 x 64] tile, 16-byte pieces ch0 .. ch0 + 3 of the row
    auto put = [&](uint8_t* dst, const float* f, int ch0) {
#pragma unroll
        for (int q8 = 0; q8 < 4; ++q8) {
            uint4 w;
            w.x = pack_bf16x2(f[q8 * 8 + 0], f[q8 * 8 + 1]); w.y = pack_bf16x2(f[q8 * 8 + 2], f[q8 * 8 + 3]);
            w.z = pack_bf16x2(f[q8 * 8 + 4], f[q8 * 8 + 5]); w.w = pack_bf16x2(f[q8 * 8 + 6], f[q8 * 8 + 7]);
            *(uint4*)(dst + trow * 128 + (((ch0 + q8) ^ sw) << 4)) = w;
        }
    };
    // this thread's 32 of the 64 channels of accumulator `col`, rotated back where they are rotary, to row trow of `out`
    auto write_rows = [&](__nv_bfloat16* out, uint32_t col, bool rotary, bool have) {
        float acc[DH / 2];
        if (have) {                                          // uniform over the CTA
            tmem_ld32(t_lane + col + hsel * 32, (uint32_t*)acc);
            tmem_ld_wait();
        } else {
#pragma unroll
            for (int i = 0; i < DH / 2; ++i) acc[i] = 0.f;
        }
        const int orow = tile * T + trow;
        if (orow >= a.l_a) return;
        if (rotary && 16 * hsel + 15 >= rope.pair0) {        // gradient w.r.t. the rotated q / k -> w.r.t. the projection
            const int pj = a.patch_idx[(size_t)pair * a.c + orow / a.l_p];
            const float t = (float)(max(pj, 0) * a.l_p + orow % a.l_p);      // (rows of unused slots are zero)
#pragma unroll
            for (int i = 0; i < DH / 4; ++i) {
                const int p = 16 * hsel + i;
                if (p < rope.pair0) continue;
                float cs, sn;
                rope_angle(rope, p, t, cs, sn);
                const float a0 = acc[2 * i], a1 = acc[2 * i + 1];
                acc[2 * i] = a0 * cs + a1 * sn;
                acc[2 * i + 1] = a1 * cs - a0 * sn;
            }
        }
        // whole sectors, two stores (in 16-byte stores, with the plan a microsecond longer: image block, training step 665.9 us, so
        // 656.7, wide block 499.7 and 494.7, language-model block 241.9 and 238.9)
        __nv_bfloat16* o = out + (size_t)(row_base + orow) * a.ld_out + col_h + hsel * 32;
        const bool whole = sector_aligned(o);
#pragma unroll
        for (int ch = 0; ch < DH / 32; ++ch) st_sector(o + 16 * ch, pack16<__nv_bfloat16>(acc + 16 * ch), pack16<__nv_bfloat16>(acc + 16 * ch + 8), whole);
    };
    auto stat = [&](const float* src, int q) { return q < a.l_a ? src[(size_t)(row_base + q) * a.heads + head] : 0.f; };
    constexpr float kLog2e = 1.4426950408889634f;

    if constexpr (MODE == kSingle) {
        uint8_t *sQ = smem, *sK = sQ + TILE_BYTES, *sV = sK + TILE_BYTES, *sDO = sV + TILE_BYTES;
        uint8_t *sP1 = sDO + TILE_BYTES, *sDS = sP1 + TILE_BYTES;            // P^T: queries 0-63 where V was, 64-127 in sP1; dS^T: two halves
        if (tid == 0) {
            mbar_arrive_expect_tx(&ctl->bar_fix, 4 * TILE_BYTES);
            tma_load_2d(sK, &m.k, col_h, row_base, &ctl->bar_fix);
            tma_load_2d(sQ, &m.q, col_h, row_base, &ctl->bar_fix);
            tma_load_2d(sV, &m.v, col_h, row_base, &ctl->bar_fix);
            tma_load_2d(sDO, &m.dout, col_h, row_base, &ctl->bar_fix);
        }
        constexpr uint32_t idesc_s = instr_desc_bf16(T, T, false, false);    // S^T = K Q^T, dP^T = V dO^T: [keys x queries]
        constexpr uint32_t idesc_k = instr_desc_bf16(T, DH, false, true);    // dV = P^T dO, dK = dS^T Q: A as written, B MN-major
        constexpr uint32_t idesc_t = instr_desc_bf16(T, DH, true, true);     // dQ = dS K: A transposed
        const uint32_t q_a = smem_u32(sQ), k_a = smem_u32(sK), v_a = smem_u32(sV), do_a = smem_u32(sDO);
        const uint32_t p1_a = smem_u32(sP1), ds_a = smem_u32(sDS);
        if (warp == 0) {
            ok = mbar_wait(&ctl->bar_fix, 0, abort_flag, status);
            __syncwarp();
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < DH / 16; ++ks)
                mma_bf16(el, tmem, smem_desc(k_a + ks * 32, 16, 1024), smem_desc(q_a + ks * 32, 16, 1024), idesc_s, ks != 0);
#pragma unroll
            for (int ks = 0; ks < DH / 16; ++ks)
                mma_bf16(el, tmem + 128, smem_desc(v_a + ks * 32, 16, 1024), smem_desc(do_a + ks * 32, 16, 1024), idesc_s, ks != 0);
            mma_commit(el, &ctl->bar_s);
        }
        // statistics of the 128 queries meanwhile: in dS's tiles, which are written only behind the barrier that follows the
        // last read of them
        float* st = (float*)sDS;                                              // [lse * log2 e | delta][128], overwritten by dS last
        if (tid < T) { st[tid] = stat(a.lse, tid) * kLog2e; st[T + tid] = stat(a.delta, tid); }
        __syncthreads();
        ok = mbar_wait(&ctl->bar_s, 0, abort_flag, status) && ok;
        const bool go = __syncthreads_and(ok && !*abort_flag);               // (uniform over the CTA)
        if (go) {
            tc_fence_after();
            // thread: key trow, queries 64 hsel .. 64 hsel + 63; dS pieces wait in registers until all statistics are read
            uint32_t ds_pk[32];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int q0 = hsel * 64 + h * 32;
                float s_v[32], dp_v[32];
                tmem_ld32(t_lane + q0, (uint32_t*)s_v);
                tmem_ld32(t_lane + 128 + q0, (uint32_t*)dp_v);
                tmem_ld_wait();
                const bool key_ok = trow < kv_end;
                p_and_ds(s_v, dp_v, a.causal ? trow - q0 : 0, key_ok ? a.l_a - q0 : 0, st + q0, st + T + q0, true);
                put(hsel == 0 ? sV : sP1, s_v, h * 4);
#pragma unroll
                for (int q = 0; q < 16; ++q) ds_pk[h * 16 + q] = pack_bf16x2(dp_v[2 * q], dp_v[2 * q + 1]);
            }
            __syncthreads();                                                  // the statistics have been read
#pragma unroll
            for (int ch = 0; ch < 8; ++ch)
                *(uint4*)(sDS + hsel * TILE_BYTES + trow * 128 + ((ch ^ sw) << 4)) =
                    make_uint4(ds_pk[4 * ch], ds_pk[4 * ch + 1], ds_pk[4 * ch + 2], ds_pk[4 * ch + 3]);
            fence_async_smem();                  // generic-proxy writes of P / dS -> visible to the tensor core
            tc_fence_before();
            __syncthreads();
            if (warp == 0) {                     // S and dP have been read: the accumulators take their columns
                tc_fence_after();
#pragma unroll
                for (int ks = 0; ks < T / 16; ++ks)
                    mma_bf16(el, tmem, smem_desc((ks < 4 ? v_a : p1_a) + (ks & 3) * 32, 16, 1024), smem_desc(do_a + ks * 2048, 8192, 1024),
                             idesc_k, ks != 0);
#pragma unroll
                for (int ks = 0; ks < T / 16; ++ks)
                    mma_bf16(el, tmem + 64, smem_desc(ds_a + (ks >> 2) * TILE_BYTES + (ks & 3) * 32, 16, 1024),
                             smem_desc(q_a + ks * 2048, 8192, 1024), idesc_k, ks != 0);
#pragma unroll
                for (int ks = 0; ks < T / 16; ++ks)
                    mma_bf16(el, tmem + 128, smem_desc(ds_a + ks * 2048, TILE_BYTES, 1024), smem_desc(k_a + ks * 2048, 8192, 1024),
                             idesc_t, ks != 0);
                mma_commit(el, &ctl->bar_o);
            }
            ok = mbar_wait(&ctl->bar_o, 0, abort_flag, status);
        }
        const bool have = __syncthreads_and(go && ok && !*abort_flag);
        tc_fence_after();
        write_rows(a.dv, 0, false, have);
        write_rows(a.dk, 64, true, have);
        write_rows(a.dq, 128, true, have);
        if (tid == 0 && *abort_flag) mbar_wait(&ctl->bar_fix, 0, abort_flag, status);      // let the copies land (bounded)
    } else {
        constexpr bool DQ = MODE == kDq;
        uint8_t *sF0 = smem, *sF1 = sF0 + TILE_BYTES;                        // resident: Q_i, dO_i | K_j, V_j
        uint8_t *sS0 = sF1 + TILE_BYTES, *sS1 = sS0 + 2 * BLK_BYTES;         // streamed: K, V | Q, dO (two stages each)
        uint8_t *sDS = sS1 + 2 * BLK_BYTES, *sP = sDS + TILE_BYTES;          // dS (dS^T); P^T (kDkDv)
        // streamed blocks [first, last]; none: the tile's output is zero
        int first = 0, last;
        if (DQ) { last = (kv_end + TS - 1) / TS - 1; if (a.causal) last = min(last, 2 * tile + 1); }
        else { last = tile * T < kv_end ? (a.l_a + TS - 1) / TS - 1 : -1; if (a.causal) first = 2 * tile; }
        const int n_it = last - first + 1;
        auto load = [&](int t) {                                             // block first + t into stage t & 1
            const int st = t & 1;
            mbar_arrive_expect_tx(&ctl->bar_ld[st], 2 * BLK_BYTES);
            tma_load_2d(sS0 + st * BLK_BYTES, tmS0, col_h, row_base + (first + t) * TS, &ctl->bar_ld[st]);
            tma_load_2d(sS1 + st * BLK_BYTES, tmS1, col_h, row_base + (first + t) * TS, &ctl->bar_ld[st]);
        };
        if (tid == 0 && n_it > 0) {
            mbar_arrive_expect_tx(&ctl->bar_fix, 2 * TILE_BYTES);
            tma_load_2d(sF0, DQ ? &m.q : &m.k, col_h, row_base + tile * T, &ctl->bar_fix);
            tma_load_2d(sF1, DQ ? &m.dout : &m.v, col_h, row_base + tile * T, &ctl->bar_fix);
            for (int t = 0; t < 2 && t < n_it; ++t) load(t);
        }
        float my_lse2 = 0.f, my_delta = 0.f;                                 // kDq: this thread's query
        auto fetch = [&](int t) {                                            // kDkDv: statistics of block first + t, a query per thread
            if (tid < TS) {
                s_stat[(t & 1) * 2 * TS + tid] = stat(a.lse, (first + t) * TS + tid) * kLog2e;
                s_stat[(t & 1) * 2 * TS + TS + tid] = stat(a.delta, (first + t) * TS + tid);
            }
        };
        if (DQ) { my_lse2 = stat(a.lse, tile * T + trow) * kLog2e; my_delta = stat(a.delta, tile * T + trow); }
        else if (n_it > 0) fetch(0);
        __syncthreads();
        constexpr uint32_t idesc_s = instr_desc_bf16(T, TS, false, false);   // S, dP (or transposed): both operands K-major
        constexpr uint32_t idesc_o = instr_desc_bf16(T, DH, false, true);    // accumulators: A as written, B MN-major
        const uint32_t f0 = smem_u32(sF0), f1 = smem_u32(sF1), ds_a = smem_u32(sDS), p_a = smem_u32(sP);

        for (int it = 0; it < n_it; ++it) {
            const int st = it & 1;
            const uint32_t s0 = smem_u32(sS0) + st * BLK_BYTES, s1 = smem_u32(sS1) + st * BLK_BYTES;
            if (warp == 0) {
                if (it == 0) ok = mbar_wait(&ctl->bar_fix, 0, abort_flag, status);
                ok = mbar_wait(&ctl->bar_ld[st], (it >> 1) & 1, abort_flag, status) && ok;
                __syncwarp();
                tc_fence_after();
#pragma unroll
                for (int ks = 0; ks < DH / 16; ++ks)
                    mma_bf16(el, tmem, smem_desc(f0 + ks * 32, 16, 1024), smem_desc(s0 + ks * 32, 16, 1024), idesc_s, ks != 0);
#pragma unroll
                for (int ks = 0; ks < DH / 16; ++ks)
                    mma_bf16(el, tmem + TS, smem_desc(f1 + ks * 32, 16, 1024), smem_desc(s1 + ks * 32, 16, 1024), idesc_s, ks != 0);
                mma_commit(el, &ctl->bar_s);
            }
            if (!DQ && it + 1 < n_it) fetch(it + 1);         // (the other stage: its readers passed the last barrier)
            ok = mbar_wait(&ctl->bar_s, it & 1, abort_flag, status) && ok;
            if (!__all_sync(0xffffffffu, ok && !*abort_flag)) ok = false;
            tc_fence_after();
            // every MMA issued before this commit has completed, the previous step's accumulation included: its stage and
            // the P / dS tiles are free again
            if (tid == 0 && it >= 1 && it + 1 < n_it && ok) load(it + 1);
            float s_v[32], dp_v[32];
            if (ok) {                                        // uniform over the warp
                tmem_ld32(t_lane + hsel * 32, (uint32_t*)s_v);
                tmem_ld32(t_lane + TS + hsel * 32, (uint32_t*)dp_v);
                tmem_ld_wait();
                const int c0 = (first + it) * TS + hsel * 32, row = tile * T + trow;     // first streamed row of the piece; resident row
                if (DQ) {
                    const int hi = row < a.l_a ? min(kv_end, a.causal ? row + 1 : kv_end) - c0 : 0;
                    p_and_ds(s_v, dp_v, 0, hi, &my_lse2, &my_delta, false);
                } else {
                    const float* sst = s_stat + st * 2 * TS + hsel * 32;
                    p_and_ds(s_v, dp_v, a.causal ? row - c0 : 0, row < kv_end ? a.l_a - c0 : 0, sst, sst + TS, true);
                    put(sP, s_v, hsel * 4);
                }
                put(sDS, dp_v, hsel * 4);
            }
            fence_async_smem();                  // generic-proxy writes of P / dS -> visible to the tensor core
            tc_fence_before();
            if (!__syncthreads_and(ok)) { ok = false; break; }
            if (warp == 0) {
                tc_fence_after();
                if (!DQ) {
#pragma unroll
                    for (int ks = 0; ks < TS / 16; ++ks)     // contraction over the 64 queries
                        mma_bf16(el, tmem + 192, smem_desc(p_a + ks * 32, 16, 1024), smem_desc(s1 + ks * 2048, 8192, 1024), idesc_o, (it | ks) != 0);
                }
#pragma unroll
                for (int ks = 0; ks < TS / 16; ++ks)
                    mma_bf16(el, tmem + 128, smem_desc(ds_a + ks * 32, 16, 1024), smem_desc(s0 + ks * 2048, 8192, 1024), idesc_o, (it | ks) != 0);
                if (it == n_it - 1) mma_commit(el, &ctl->bar_o);
            }
        }
        bool have = n_it > 0 && ok;
        if (have) have = mbar_wait(&ctl->bar_o, 0, abort_flag, status) && !*abort_flag;
        have = __syncthreads_and(have);
        tc_fence_after();
        write_rows(DQ ? a.dq : a.dk, 128, true, have);
        if (!DQ) write_rows(a.dv, 192, false, have);
        if (tid == 0 && *abort_flag && n_it > 0) {           // let copies that may still be in flight land (bounded)
            mbar_wait(&ctl->bar_fix, 0, abort_flag, status);
            for (int t = 0; t < 2 && t < n_it; ++t) mbar_try_wait(&ctl->bar_ld[t], 0);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        tmem_dealloc(tmem, 256);
    }
}

// one tile of 128 tokens per pair; grid (heads, pairs)
__global__ void __launch_bounds__(kThreads, 2)
attn_bwd_single_kernel(const __grid_constant__ BwdMaps m, const __grid_constant__ BwdArgs a,
                       const __grid_constant__ Rope rope /* pair0 < 32: dq and dk are rotated back (Eq. 32) */) {
    pdl_trigger();
    attn_bwd_body<kSingle>(m, m, a, rope, 0);
}

// grid (heads, pairs, 2 n_tiles): key tiles and query tiles in one launch, longest streams first (low key tiles see the most
// queries, high query tiles the most keys)
__global__ void __launch_bounds__(kThreads, 2)
attn_bwd_stream_kernel(const __grid_constant__ BwdMaps m, const __grid_constant__ BwdMaps mb, const __grid_constant__ BwdArgs a,
                       const __grid_constant__ Rope rope) {
    pdl_trigger();
    const int z = blockIdx.z;
    if (z & 1) attn_bwd_body<kDq>(m, mb, a, rope, a.n_tiles - 1 - z / 2);
    else attn_bwd_body<kDkDv>(m, mb, a, rope, z / 2);
}

}  // namespace

// q, k, v, dout: [rows_max, d_g] bf16 routed buffers; dq, dk, dv: bf16 with ld_out elements per row;
// lse, delta: [rows_max, heads] float32 (lse as written by the forward kernel, natural logarithm).
uoe_status launch_attention_backward(const Dims& D, const void* q, const void* k, const void* v, const void* dout,
                                     const float* lse, const float* delta, void* dq, void* dk, void* dv, int ld_out,
                                     const int* pair_row, const int* patch_idx, bool causal, const Rope& rope, int* status,
                                     cudaStream_t s) {
    if (D.d_h != DH) return UOE_ERR_UNSUPPORTED;
    static SpreadOnce once[2];
    {
        uoe_status st = smem_opt_in(once[0].opt_in, attn_bwd_single_kernel, 160 * 1024);
        if (st == UOE_OK) st = smem_opt_in(once[1].opt_in, attn_bwd_stream_kernel, 160 * 1024);
        if (st != UOE_OK) return st;
    }
    const int heads = D.d_g / DH, n_tiles = (D.l_a + T - 1) / T;
    const long long pairs = (long long)D.B * D.k;
    if (pairs > 65535 || 2 * n_tiles > 65535) return UOE_ERR_UNSUPPORTED;      // pairs ride on grid.y, tiles on grid.z
    BwdMaps m, mb;                                // [128 x 64] tiles and [64 x 64] blocks of q, k, v, dout
    const void* ptrs[4] = {q, k, v, dout};
    CUtensorMap* maps[2][4] = {{&m.q, &m.k, &m.v, &m.dout}, {&mb.q, &mb.k, &mb.v, &mb.dout}};
    for (int i = 0; i < 4; ++i) {
        const uint64_t dims[2] = {(uint64_t)D.d_g, (uint64_t)D.Rmax};
        const uint64_t str[1] = {(uint64_t)D.d_g * 2};
        const uint32_t box[2] = {DH, T}, box_s[2] = {DH, TS};
        if (!make_tmap(maps[0][i], ptrs[i], 2, dims, str, box) || !make_tmap(maps[1][i], ptrs[i], 2, dims, str, box_s)) return UOE_ERR_CUDA;
    }
    BwdArgs a;
    a.dq = (__nv_bfloat16*)dq; a.dk = (__nv_bfloat16*)dk; a.dv = (__nv_bfloat16*)dv; a.ld_out = ld_out;
    a.lse = lse; a.delta = delta; a.pair_row = pair_row; a.patch_idx = patch_idx;
    a.c = D.c; a.l_p = D.l_p; a.Lv = D.Lv; a.l_a = D.l_a; a.heads = heads; a.causal = causal ? 1 : 0; a.n_tiles = n_tiles;
    a.scale_log2 = 1.4426950408889634f / sqrtf((float)D.d_h);
    a.inv_sqrt_dh = 1.0f / sqrtf((float)D.d_h);
    a.status = status;
    ProfScope ps("attn_bwd", s);
    if (n_tiles == 1) {
        launch_k(attn_bwd_single_kernel, dim3(heads, (unsigned)pairs), dim3(kThreads),
                 spread_smem(once[0], attn_bwd_single_kernel, pairs * heads, BCfg<kSingle>::SMEM), s, m, a, rope);
    } else {
        launch_k(attn_bwd_stream_kernel, dim3(heads, (unsigned)pairs, 2 * n_tiles), dim3(kThreads),
                 spread_smem(once[1], attn_bwd_stream_kernel, 2 * pairs * heads * n_tiles, BCfg<kDkDv>::SMEM), s, m, mb, a, rope);
    }
    UOE_LAUNCHED();
    return UOE_OK;
}

}  // namespace uoe
