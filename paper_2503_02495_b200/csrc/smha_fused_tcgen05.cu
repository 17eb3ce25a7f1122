// Projections and attention in one kernel (Eq. 28-35) for experts of one 64-wide head whose pairs have few tokens: a CTA takes
// 128 queries of one (sample, chosen expert) pair from x to z = softmax(q k^T / sqrt(d_h) + mask) v W^o, so that q (and, with one
// tile of queries, k and v) never leave the SM and a launch with its hand-over falls away.
//
//   warp 8      TMA producer: A [128 x 64] gathered from x (Eq. 18, one box per source patch) and [64 x 64] blocks of W^q, W^k,
//               W^v per K step through a ring; then key tiles and W^o in 128-column chunks
//   warp 9      MMA issuer: q | k | v [128 x 192] into TMEM, S = q k^T, O_t = P v, z chunks = o W^o
//   warps 0-7   q, k, v -> (rotary positions) -> bf16 tiles in shared memory where the ring was; softmax with two threads per
//               query row; o -> bf16 tile; z chunks -> memory
//
// MULTI = false: pairs of at most 128 tokens, one CTA each, all operands of the attention in the CTA's own shared memory; two CTAs
// per SM (80 KB of ring, 256 TMEM columns), one's loads and products under the other's exponentials and write-out.
// MULTI = true: pairs of two to eight full tiles, a cluster of as many CTAs, one CTA per SM with a longer ring.  Every CTA
// projects its own tile, stores its k and v (they stay in L2), works on its own keys, and streams the other tiles once every CTA of
// the cluster has arrived at its barrier.
//
// With `q` set the kernel is the backward's recomputation instead: q, k, v, o and the log-sum-exp are written, z is not.
#include "attn_out.cuh"
#include "hand_over.h"
#include "kernels.cuh"
#include "tc.cuh"
#include "tmap.cuh"

#include <type_traits>

namespace uoe {
namespace {

using namespace tc;

constexpr int T = 128, DH = 64, BK = 64;
constexpr int UNIT = 16384;                              // a [128 x 64] bf16 tile
constexpr int STAGE = UNIT + 3 * 8192;                   // A and a block of each of the three weights
constexpr int kSoftWarps = 8, kThreads = 32 * (kSoftWarps + 2);
constexpr int ZC = 128;                                  // output columns of a z chunk

template <bool MULTI> struct FCfg {
    static constexpr int STAGES = MULTI ? 5 : 2;
    // after the projection the ring's place holds, in units of a tile:  q, then
    //   single: k, v, P (two halves; o in the first), a chunk of W^o from the start; later two more where q and k were
    //   multi:  P (the same), two key stages (k | v), own k, v, two W^o chunks, z staging (two); later two more chunks where own k
    //           and v were
    static constexpr int K = MULTI ? 7 : 1, V = MULTI ? 8 : 2, P = MULTI ? 1 : 3, KV = 3;
    static constexpr int NW = MULTI ? 4 : 3;             // W^o chunks held
    __host__ __device__ static constexpr int W(int b) { return MULTI ? (b < 2 ? 9 + b : 5 + b) : (b == 0 ? 5 : b - 1); }
    static constexpr int UNITS = MULTI ? 13 : 6;
    static constexpr int TMEM = MULTI ? 512 : 256;       // q k v [0, 192); S [0, 128) (multi: and [128, 256)); O; z chunks [0, 256)
    static constexpr int COL_O = MULTI ? 256 : 128;
    static constexpr int SMEM = UNITS * UNIT + 1024 /*alignment*/ + 512 /*control*/;
};
static_assert(FCfg<false>::STAGES * STAGE <= FCfg<false>::W(0) * UNIT && FCfg<true>::STAGES * STAGE <= FCfg<true>::UNITS * UNIT, "ring");
static_assert(2 * (FCfg<false>::SMEM + 2048 + 1024) <= 228 * 1024, "two CTAs per SM");

struct FuCtl {
    uint64_t full[5], empty[5], qkv_full, qkv_ready /* multi */, kv_full[2], kv_empty[2], s_full, o_full, own_free, w_full[4], w_empty[4],
        z_full[2], z_free[2];
    uint32_t tmem_base;
    int abort_flag, n_valid, pad;
};
static_assert(sizeof(FuCtl) <= 512, "control block");

struct FuMaps { CUtensorMap x, w[3], k, v, wo, z; };

struct FuArgs {
    __nv_bfloat16 *q, *k, *v, *o;       // [rows, 64]; q null: forward
    __nv_bfloat16* z;                   // [rows, d], forward
    float* lse;                         // [rows] or null
    const int *pair_row, *patch_idx, *expert_idx, *expert_end, *offsets;
    int pairs, n, m, k_sel, c, lp_log, Lv, l_a, d, causal, n_qt;
    float scale_log2;
    int* status;
};

// Hand-over p from the softmax warps to the MMA warp, by the rule of hand_over.h: they arrive, it waits, on a barrier of the SM, which
// wakes it sooner than an mbarrier does (image block forward 190.3 us through mbarriers, 187.6 so; language-model block 69.5 and 69.0).
constexpr int kHandOver = 6;              // and 7
__device__ __forceinline__ void hand_over_wait(int p) { hand_over_take<32 * (kSoftWarps + 1)>(kHandOver + hand_over_barrier(p)); }
__device__ __forceinline__ void hand_over_arrive(int p, bool ok) { hand_over_write<32 * (kSoftWarps + 1)>(kHandOver + hand_over_barrier(p), !ok); }
__device__ __forceinline__ void bar_named(int id, int threads) { asm volatile("bar.sync %0, %1;" :: "r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void fence_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

struct NoRopeF {};

template <bool MULTI, bool ROPE>
__global__ void __launch_bounds__(kThreads, MULTI ? 1 : 2)
smha_fused_kernel(const __grid_constant__ FuMaps tm, const FuArgs a,
                  const __grid_constant__ typename std::conditional<ROPE, Rope, NoRopeF>::type rope) {
    using Cf = FCfg<MULTI>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    FuCtl* ctl = (FuCtl*)(smem + Cf::UNITS * UNIT);
    __shared__ float s_xch[2][T];                        // per row: the two halves' maxima, later their sums
    volatile int* abort_flag = &ctl->abort_flag;
    int* status = a.status;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int pair = (int)blockIdx.x / a.n_qt, qt = (int)blockIdx.x - pair * a.n_qt;
    const int q0 = qt * T, l_p = 1 << a.lp_log;
    auto unit = [&](int u) { return smem + u * UNIT; };

    if (tid == 0) {
        for (int s = 0; s < Cf::STAGES; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 1); }
        mbar_init(&ctl->qkv_full, 1);
        mbar_init(&ctl->qkv_ready, 32 * kSoftWarps);
        for (int s = 0; s < 2; ++s) {
            mbar_init(&ctl->kv_full[s], 1); mbar_init(&ctl->kv_empty[s], 1);
            mbar_init(&ctl->z_full[s], 1); mbar_init(&ctl->z_free[s], 32 * kSoftWarps);
        }
        for (int s = 0; s < Cf::NW; ++s) { mbar_init(&ctl->w_full[s], 1); mbar_init(&ctl->w_empty[s], 1); }
        mbar_init(&ctl->own_free, 1);
        mbar_init(&ctl->s_full, 1);
        mbar_init(&ctl->o_full, 1);
        ctl->abort_flag = 0;
        fence_barrier_init();
        prefetch_tmap(&tm.x);
        prefetch_tmap(&tm.w[0]); prefetch_tmap(&tm.w[1]); prefetch_tmap(&tm.w[2]);
    }
    if (warp == 9) {
        tmem_alloc(&ctl->tmem_base, Cf::TMEM);
        pdl_trigger();          // only now: a CTA of a later kernel that fits beside this one must not take its columns and then wait for it
    }
    pdl_wait();                                          // from here on: data written by earlier kernels
    const int expert = a.expert_idx[pair];
    const bool named = (unsigned)expert < (unsigned)a.n; // (a caller's slot that names no expert has been reported; nothing is written for it)
    const int row_base = a.pair_row[pair];
    int my_src = a.pairs / a.k_sel * a.m;                // source patch of this lane's box; past the last patch: zero rows
    if (warp == 8) {
        int nv = 0;                                      // real keys of the pair
        for (int u = lane; u < a.c; u += 32) {
            const int j = a.patch_idx[(size_t)pair * a.c + u];
            if (j >= 0) nv += max(0, min(l_p, a.Lv - j * l_p));
        }
        nv = __reduce_add_sync(0xffffffffu, nv);
        if (lane == 0) ctl->n_valid = named ? nv : 0;
        const int u = (q0 >> a.lp_log) + lane;
        if (lane < (T >> a.lp_log) && u < a.c) {
            const int j = a.patch_idx[(size_t)pair * a.c + u];
            if (j >= 0 && j < a.m) my_src = pair / a.k_sel * a.m + j;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    int kv_end = min(ctl->n_valid, a.l_a);
    if (a.causal) kv_end = min(kv_end, q0 + T);
    const int n_kv = (kv_end + T - 1) / T;               // key tiles of this CTA's queries; 0 for a pair without a patch
    // multi: the CTA's own tile first (it is in shared memory, the others are on their way), then the others in order.  (In
    // ascending order, as in the separate kernels, the own tile waits for the others': one sequence 54.6 us, so 52.9, language-model block
    // 66.7 and 64.4, its training step 227.8 and 223.6.  The sums round in another order: gradients move by up to 8e-4 of their norm,
    // the distance of dW_q, dW_k, dW_v, dW_o from float64, 2.8e-3 to 3.7e-3, by less than 0.1 %, that of dW_r, 2.6e-3 to 2.8e-3, by
    // -2.3 to +0.5 %.)
    const bool own = !MULTI || qt < n_kv;
    auto tile_at = [&](int i) { return !MULTI ? 0 : (!own ? i : (i == 0 ? qt : (i - 1 < qt ? i - 1 : i))); };
    const int num_kb = a.d / BK;
    const bool keep = a.q != nullptr;                    // the backward's recomputation
    const int n_z = keep || n_kv == 0 ? 0 : (a.d + ZC - 1) / ZC;
    auto wait = [&](uint64_t* bar, uint32_t parity) { return mbar_wait(bar, parity, abort_flag, status) && !*abort_flag; };

    if (warp == 8) {
        // =========================== TMA producer ===========================
        bool ok = true;
        int issued = 0, kv_issued = 0, w_issued = 0;
        for (int kb = 0; kb < num_kb && ok; ++kb) {
            const int st = kb % Cf::STAGES;
            int w = 1;
            if (lane == 0) {
                w = wait(&ctl->empty[st], ((kb / Cf::STAGES) & 1) ^ 1) ? 1 : 0;
                if (w) mbar_arrive_expect_tx(&ctl->full[st], STAGE);
            }
            ok = __shfl_sync(0xffffffffu, w, 0) != 0;
            if (!ok) break;
            uint8_t* sa = smem + st * STAGE;
            if (lane < (T >> a.lp_log)) tma_load_3d(sa + (lane << a.lp_log) * 128, &tm.x, kb * BK, 0, my_src, &ctl->full[st]);
            if (lane < 3) tma_load_4d(sa + UNIT + lane * 8192, &tm.w[lane], 0, kb * BK, 0, expert, &ctl->full[st]);
            ++issued;
        }
        auto load_w = [&]() {                            // the next chunk of W^o
            const int j = w_issued, st = j % Cf::NW, nn = min(ZC, a.d - j * ZC);
            if (!wait(&ctl->w_empty[st], ((j / Cf::NW) & 1) ^ 1)) return false;
            mbar_arrive_expect_tx(&ctl->w_full[st], (uint32_t)nn * DH * 2);
            for (int nb = 0; nb < nn / 64; ++nb) tma_load_3d(unit(Cf::W(st)) + nb * 8192, &tm.wo, j * ZC + nb * 64, 0, expert, &ctl->w_full[st]);
            ++w_issued;
            return true;
        };
        if constexpr (MULTI) {
            if (lane == 0) {                             // own k and v to memory
                ok = ok && wait(&ctl->qkv_ready, 0);
                if (ok && named) {
                    tma_store_2d(&tm.k, unit(Cf::K), 0, row_base + q0);
                    tma_store_2d(&tm.v, unit(Cf::V), 0, row_base + q0);
                    bulk_commit();
                    for (int j = 0; j < 2 && j < n_z && ok; ++j) ok = load_w();
                    bulk_wait_all();
                    fence_async_all();
                }
            }
            __syncwarp();
            cluster_sync_all();                          // every CTA's are there
            if (lane == 0 && ok) {
                fence_async_all();
                for (int i = own ? 1 : 0; i < n_kv && ok; ++i) {
                    const int q = kv_issued, st = q & 1, t = tile_at(i);
                    ok = wait(&ctl->kv_empty[st], ((q >> 1) & 1) ^ 1);
                    if (!ok) break;
                    mbar_arrive_expect_tx(&ctl->kv_full[st], 2 * UNIT);
                    tma_load_2d(unit(Cf::KV + 2 * st), &tm.k, 0, row_base + t * T, &ctl->kv_full[st]);
                    tma_load_2d(unit(Cf::KV + 2 * st + 1), &tm.v, 0, row_base + t * T, &ctl->kv_full[st]);
                    ++kv_issued;
                }
                if (w_issued < n_z && own) ok = ok && wait(&ctl->own_free, 0);
            }
        } else if (lane == 0 && ok && n_z > 0) {
            ok = load_w();
            ok = ok && wait(&ctl->s_full, 0);           // S is done: q and k may be overwritten
        }
        if (lane == 0)
            while (ok && w_issued < n_z) ok = load_w();
        if (lane == 0 && *abort_flag) {                  // let copies that may still be in flight land (bounded)
            for (int t = max(0, issued - Cf::STAGES); t < issued; ++t) mbar_wait(&ctl->full[t % Cf::STAGES], (t / Cf::STAGES) & 1, abort_flag, status);
            for (int t = max(0, kv_issued - 2); t < kv_issued; ++t) mbar_wait(&ctl->kv_full[t & 1], (t >> 1) & 1, abort_flag, status);
            for (int t = max(0, w_issued - Cf::NW); t < w_issued; ++t) mbar_wait(&ctl->w_full[t % Cf::NW], (t / Cf::NW) & 1, abort_flag, status);
        }
        __syncwarp();
    } else if (warp == 9) {
        // =========================== MMA issuer (the whole warp, one elected lane issues) ===========================
        const uint32_t el = elect_one();
        auto waitw = [&](uint64_t* bar, uint32_t parity) { return __all_sync(0xffffffffu, wait(bar, parity)) != 0; };
        constexpr uint32_t idesc_p = instr_desc_bf16(T, 192, false, true), idesc_s = instr_desc_bf16(T, T, false, false);
        constexpr uint32_t idesc_o = instr_desc_bf16(T, DH, false, true);
        bool ok = true;
        for (int kb = 0; kb < num_kb && ok; ++kb) {
            const int st = kb % Cf::STAGES;
            ok = waitw(&ctl->full[st], (kb / Cf::STAGES) & 1);
            if (!ok) break;
            tc_fence_after();
            const uint32_t sa = smem_u32(smem + st * STAGE), sb = sa + UNIT;
#pragma unroll
            for (int ks = 0; ks < BK / 16; ++ks)
                mma_bf16(el, tmem, smem_desc(sa + ks * 32, 16, 1024), smem_desc(sb + ks * 2048, 8192, 1024), idesc_p, (kb | ks) != 0);
            mma_commit(el, &ctl->empty[st]);
        }
        if (ok) mma_commit(el, &ctl->qkv_full);
        if constexpr (MULTI) cluster_arrive();
        hand_over_wait(0);                               // q, k, v are in shared memory
        const uint32_t qa = smem_u32(unit(0)), pa = smem_u32(unit(Cf::P));
        // place of the i-th tile's k and v: own, or stage q & 1 of the others
        auto stage_of = [&](int i) { return own ? i - 1 : i; };
        auto issue_s = [&](int i) {
            const int q = stage_of(i);
            if (MULTI && q >= 0 && !waitw(&ctl->kv_full[q & 1], (q >> 1) & 1)) return false;
            tc_fence_after();
            const uint32_t ka = smem_u32(MULTI && q >= 0 ? unit(Cf::KV + 2 * (q & 1)) : unit(Cf::K));
#pragma unroll
            for (int ks = 0; ks < DH / 16; ++ks)
                mma_bf16(el, tmem + (MULTI ? (i & 1) * T : 0), smem_desc(qa + ks * 32, 16, 1024), smem_desc(ka + ks * 32, 16, 1024), idesc_s, ks != 0);
            mma_commit(el, &ctl->s_full);
            return true;
        };
        if (n_kv > 0) ok = ok && issue_s(0);
        for (int i = 0; i < n_kv; ++i) {
            hand_over_wait(MULTI ? 1 + i : 1);           // P is
            ok = __all_sync(0xffffffffu, ok && !*abort_flag) != 0;
            if (!ok) continue;
            tc_fence_after();
            const int q = stage_of(i);
            const uint32_t va = smem_u32(MULTI && q >= 0 ? unit(Cf::KV + 2 * (q & 1) + 1) : unit(Cf::V));
#pragma unroll
            for (int ks = 0; ks < T / 16; ++ks)
                mma_bf16(el, tmem + Cf::COL_O, smem_desc(pa + (ks >> 2) * UNIT + (ks & 3) * 32, 16, 1024), smem_desc(va + ks * 2048, 8192, 1024),
                         idesc_o, ks != 0);
            mma_commit(el, &ctl->o_full);
            if (MULTI) mma_commit(el, q >= 0 ? &ctl->kv_empty[q & 1] : &ctl->own_free);
            if (i + 1 < n_kv) ok = issue_s(i + 1);       // (into the other accumulator: it runs under the O update)
        }
        if (n_kv > 0) hand_over_wait(MULTI ? 1 + n_kv : 2);      // o is
        ok = __all_sync(0xffffffffu, ok && !*abort_flag) != 0;
        for (int j = 0; j < n_z && ok; ++j) {
            const int st = j & 1, wb = j % Cf::NW;
            ok = waitw(&ctl->w_full[wb], (j / Cf::NW) & 1) && waitw(&ctl->z_free[st], ((j >> 1) & 1) ^ 1);
            if (!ok) break;
            tc_fence_after();
            const uint32_t wa = smem_u32(unit(Cf::W(wb))), idesc_z = instr_desc_bf16(T, min(ZC, a.d - j * ZC), false, true);
#pragma unroll
            for (int ks = 0; ks < DH / 16; ++ks)
                mma_bf16(el, tmem + st * ZC, smem_desc(pa + ks * 32, 16, 1024), smem_desc(wa + ks * 2048, 8192, 1024), idesc_z, ks != 0);
            mma_commit(el, &ctl->z_full[st]);
            mma_commit(el, &ctl->w_empty[wb]);
        }
    } else {
        // =========================== softmax warps ===========================
        // (a wait that runs out leaves ok false: the work is skipped, the hand-overs and the barriers of CTA and cluster are not)
        const int quarter = warp & 3, hsel = warp >> 2;  // TMEM lane quarter; half of the columns
        const int trow = quarter * 32 + lane, qrow = q0 + trow, sw = trow & 7;
        const uint32_t t_lane = tmem + ((uint32_t)(quarter * 32) << 16);
        const int left = a.l_a - (q0 + quarter * 32);    // rows of the pair from this quarter's first on
        auto put = [&](uint8_t* tile, const float* f, int ch0) {     // 32 columns of this thread's row, 16-byte pieces ch0 ..
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint4 w;
                w.x = pack_bf16x2(f[8 * c + 0], f[8 * c + 1]); w.y = pack_bf16x2(f[8 * c + 2], f[8 * c + 3]);
                w.z = pack_bf16x2(f[8 * c + 4], f[8 * c + 5]); w.w = pack_bf16x2(f[8 * c + 6], f[8 * c + 7]);
                *(uint4*)(tile + trow * 128 + (((ch0 + c) ^ sw) << 4)) = w;
            }
        };
        // this quarter's valid rows of a tile to rows of [rows, 64], half of them per warp (both warps have written theirs)
        auto copy_out = [&](const uint8_t* tile, __nv_bfloat16* out) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = hsel * 16 + i * 4 + (lane >> 3), ch = lane & 7, tr = quarter * 32 + r;
                if (r < left) *(uint4*)(out + (size_t)(row_base + q0 + tr) * DH + ch * 8) = *(const uint4*)(tile + tr * 128 + ((ch ^ (tr & 7)) << 4));
            }
        };
        int tok = 0;                                     // position of this thread's row in its sample
        if constexpr (ROPE) {
            const int u = qrow >> a.lp_log;
            const int pj = u < a.c ? a.patch_idx[(size_t)pair * a.c + u] : -1;
            tok = pj >= 0 ? (pj << a.lp_log) + (qrow & (l_p - 1)) : 0;
        }
        // a warp takes the same 32 channels of q and of k: their angles once, under the projection's products
        [[maybe_unused]] float cs[16], sn[16];
        if constexpr (ROPE) {
#pragma unroll
            for (int p = 0; p < 16; ++p) {
                cs[p] = 1.f;
                sn[p] = 0.f;
                if (hsel * 16 + p >= rope.pair0) rope_angle(rope, hsel * 16 + p, (float)tok, cs[p], sn[p]);
            }
        }
        if (keep) {                                      // padding rows of the expert regions: zeros, as tiles may reach over them
            for (int e = blockIdx.x; e < a.n; e += gridDim.x) {
                const int r0 = a.expert_end[e], vecs = (a.offsets[e + 1] - r0) * (DH / 8);
                for (int i = tid; i < vecs; i += 32 * kSoftWarps) {
                    const uint4 zero = make_uint4(0, 0, 0, 0);
                    const size_t at = (size_t)r0 * (DH / 8) + i;
                    ((uint4*)a.q)[at] = zero; ((uint4*)a.k)[at] = zero; ((uint4*)a.v)[at] = zero;
                }
            }
        }
        // ---- q, k, v: bf16 tiles (K-major for q and k, MN-major for v: the same layout) ----
        bool ok = __all_sync(0xffffffffu, wait(&ctl->qkv_full, 0)) != 0;
        if (ok) {
            tc_fence_after();
#pragma unroll
            for (int g = 0; g < 3; ++g) {
                float f[32];
                tmem_ld32(t_lane + g * DH + hsel * 32, (uint32_t*)f);
                tmem_ld_wait();
                if constexpr (ROPE) {
                    if (g < 2) {
#pragma unroll
                        for (int p = 0; p < 16; ++p) {   // Eq. 32 on the float32 accumulators
                            const float x0 = f[2 * p], x1 = f[2 * p + 1];
                            f[2 * p] = x0 * cs[p] - x1 * sn[p];
                            f[2 * p + 1] = x0 * sn[p] + x1 * cs[p];
                        }
                    }
                }
                put(unit(g == 0 ? 0 : (g == 1 ? Cf::K : Cf::V)), f, hsel * 4);
            }
            fence_async_smem();
            tc_fence_before();
            if (MULTI) mbar_arrive(&ctl->qkv_ready);
        }
        hand_over_arrive(0, ok);
        if constexpr (MULTI) cluster_arrive();
        if (keep) {
            bar_named(2 + quarter, 64);
            if (ok && named) {
                copy_out(unit(0), a.q);
                if (!MULTI) { copy_out(unit(Cf::K), a.k); copy_out(unit(Cf::V), a.v); }
            }
        }

        // ---- online softmax over the key tiles ----
        constexpr int HK = T / 2, HD = DH / 2;
        float o_acc[HD];
#pragma unroll
        for (int i = 0; i < HD; ++i) o_acc[i] = 0.f;
        float m_run = -INFINITY, l_run = 0.f;            // l_run: sum over this thread's half of the keys
        const int kv_lim = min(ctl->n_valid, a.l_a);
        for (int i = 0; i < n_kv; ++i) {
            const int t = tile_at(i);
            ok = ok && __all_sync(0xffffffffu, wait(&ctl->s_full, i & 1)) != 0;
            float s[HK], m_new = m_run;
            const int keep_cols = min(kv_lim, a.causal ? qrow + 1 : kv_lim) - t * T - hsel * HK;
            if (ok) {
                tc_fence_after();
                tmem_ld32(t_lane + (MULTI ? (i & 1) * T : 0) + hsel * HK, (uint32_t*)s);
                tmem_ld32(t_lane + (MULTI ? (i & 1) * T : 0) + hsel * HK + 32, (uint32_t*)(s + 32));
                tmem_ld_wait();
                if (t * T + T > kv_lim || (a.causal && t * T + T - 1 > q0)) {
#pragma unroll
                    for (int j = 0; j < HK; ++j) {
                        s[j] = j < keep_cols ? s[j] * a.scale_log2 : -INFINITY;
                        m_new = fmaxf(m_new, s[j]);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < HK; ++j) {
                        s[j] *= a.scale_log2;
                        m_new = fmaxf(m_new, s[j]);
                    }
                }
            }
            s_xch[hsel][trow] = m_new;                   // (the tile before: read by everybody before its P was complete)
            bar_named(2 + quarter, 64);
            m_new = fmaxf(m_new, s_xch[hsel ^ 1][trow]);
            const float m_use = (m_new == -INFINITY) ? 0.f : m_new;          // a row with no kept key so far
            const float alpha = ex2_approx(m_run - m_use);
            if (ok) {
                float l_add = 0.f;
                uint8_t* tile = unit(Cf::P + hsel);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) { s[h * 32 + j] = ex2_approx(s[h * 32 + j] - m_use); l_add += s[h * 32 + j]; }
                    put(tile, s + h * 32, h * 4);
                }
                l_run = l_run * alpha + l_add;
                m_run = m_new;
                fence_async_smem();
                tc_fence_before();
            }
            hand_over_arrive(MULTI ? 1 + i : 1, ok);
            ok = ok && __all_sync(0xffffffffu, wait(&ctl->o_full, i & 1)) != 0;
            if (ok) {
                tc_fence_after();
                float o_t[HD];
                tmem_ld32(t_lane + Cf::COL_O + hsel * HD, (uint32_t*)o_t);
                tmem_ld_wait();
#pragma unroll
                for (int c = 0; c < HD; ++c) o_acc[c] = MULTI ? o_acc[c] * alpha + o_t[c] : o_t[c];
                tc_fence_before();
            }
            if (!MULTI) break;                           // one key tile at most
        }
        if (n_kv > 0) {
            s_xch[hsel][trow] = l_run;
            bar_named(2 + quarter, 64);
            l_run += s_xch[hsel ^ 1][trow];
            const float inv = l_run > 0.f ? 1.0f / l_run : 0.f;
            if (ok && a.lse && hsel == 0 && qrow < a.l_a) a.lse[row_base + qrow] = (m_run + log2f(l_run)) * 0.69314718055994531f;
            if (ok) {
#pragma unroll
                for (int i = 0; i < HD; ++i) o_acc[i] *= inv;
                put(unit(Cf::P), o_acc, hsel * 4);       // o [128 x 64] where the first half of P was
                fence_async_smem();
                tc_fence_before();
            }
            hand_over_arrive(MULTI ? 1 + n_kv : 2, ok);
            if (keep) {
                bar_named(2 + quarter, 64);
                if (ok) copy_out(unit(Cf::P), a.o);
            }
        } else if (a.lse && named && hsel == 0 && qrow < a.l_a) {
            a.lse[row_base + qrow] = -INFINITY;          // a pair without a key
        }
        // ---- z = o W^o_i (Eq. 35), a chunk's 64-column groups dealt to the two warps of a lane quarter ----
        [[maybe_unused]] uint8_t* stg = MULTI ? unit(11 + hsel) + quarter * 4096 : nullptr;
        for (int j = 0; j < n_z && ok; ++j) {
            const int st = j & 1, col = j * ZC + hsel * 64;
            ok = __all_sync(0xffffffffu, wait(&ctl->z_full[st], (j >> 1) & 1)) != 0;
            if (!ok) break;
            tc_fence_after();
            float zf[64];
            if (col < a.d) {                             // (uniform over the warp)
                tmem_ld32(t_lane + st * ZC + hsel * 64, (uint32_t*)zf);
                tmem_ld32(t_lane + st * ZC + hsel * 64 + 32, (uint32_t*)(zf + 32));
                tmem_ld_wait();
            }
            tc_fence_before();
            mbar_arrive(&ctl->z_free[st]);
            if (col < a.d) {
                if constexpr (MULTI) store_z_piece(zf, stg, &tm.z, a.z, a.d, col, row_base + q0 + quarter * 32, left, lane);
                else store_z_direct(zf, a.z, a.d, col, row_base + q0 + quarter * 32, left, lane);
            }
        }
        if (MULTI && lane == 0) bulk_wait_all();         // this warp's tensor stores are complete
    }
    if constexpr (MULTI) {
        if (warp != 8) cluster_wait();                   // (long complete: every thread that arrives waits)
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 9) {
        __syncwarp();
        tmem_dealloc(tmem, Cf::TMEM);
    }
}

template <bool MULTI, bool ROPE>
struct FuLaunch {
    static auto kernel() { return smha_fused_kernel<MULTI, ROPE>; }
    static uoe_status opt_in() {
        static DeviceOnce once;
        return smem_opt_in(once, kernel(), FCfg<MULTI>::SMEM);
    }
};

// How many clusters of `size` CTAs of the multi-tile kernel the current device holds at once.
int resident_clusters(int size) {
    static DeviceValue cache[9];
    const int dev = current_device();
    if (dev < 0) return 0;
    if (!cache[size].has(dev)) {
        if (FuLaunch<true, false>::opt_in() != UOE_OK) return 0;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        cfg.gridDim = dim3(size);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = FCfg<true>::SMEM;
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)size; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int v = 0;
        if (cudaOccupancyMaxActiveClusters(&v, FuLaunch<true, false>::kernel(), &cfg) != cudaSuccess) { cudaGetLastError(); v = 0; }
        cache[size].set(dev, v);
    }
    return cache[size].get(dev);
}

}  // namespace

bool smha_can_fuse(const Dims& D, bool recompute) {
    if (!can_fuse_gather(D) || D.d_h != DH || D.d_g != DH || D.n > 31) return false;
    // Forward: widths up to 512, where the kernel was made.  Beyond, block forward, one kernel / separate: d = 576 71.1 / 74.2 us (64 pairs
    // of 128 tokens), 286 / 318 (600), 80.4 / 90.2 (64 causal pairs of 256); d = 640 73.1 / 76.8, 276 / 296, 80.5 / 88.0; d = 1024 89.2 / 85.9,
    // 398 / 409, 93.8 / 101.3: the line could lie higher except for few pairs of one tile, whose CTAs have a long projection to themselves.
    if (!recompute && D.d > 512) return false;
    const int n_qt = (D.l_a + T - 1) / T;
    const long long pairs = (long long)D.B * D.k;
    // One tile: always while all pairs are resident at once, which leaves the launch in between as pure gain (400 pairs of 16 / 48 tokens,
    // d = 512: block forward 82.0 / 97.6 us, separate launches 88.1 / 110.5).  Beyond that short pairs cost: a CTA projects 128 rows
    // whatever they hold, the grouped projection packs them.  Block forward, d = 512, one kernel / separate: pairs of 48 tokens 122 / 132 us
    // (600 of them), 312 / 334 (2000); of 32 tokens 117 / 124.5 (600), 184 / 193 (1200), 269 / 279 (2000); of 16 tokens 97.5 / 102.6 (600),
    // 158 / 164 (1200), 211 / 210 (2000); d = 256, 4000 pairs of 32 tokens 203 / 202.  So the lines at 48 tokens and at four pairs per SM
    // are on the safe side: up to 2000 pairs of 16 tokens and more of 32 the one kernel would still gain 2 to 6 %.
    // The recomputation also writes q, k, v, o.  Training step, d = 512, one kernel / separate: 1600 pairs of 16 / 48 / 80 tokens 548 / 522,
    // 788 / 776, 1019 / 1014 us, 300 pairs 238 / 236, 259 / 255, 309 / 311; backward of 4000 pairs of 80 / 96 tokens 971 / 952, 1120 / 1133.
    if (n_qt == 1) {
        if (pairs <= 2ll * sm_count()) return true;
        if (recompute) return D.l_a >= 96;
        return D.l_a >= 48 || pairs <= 4ll * sm_count();
    }
    // Several tiles: while all clusters are resident at once (16 causal pairs of 256 tokens, d = 512: forward 25.2 us, separate
    // launches 28.7; two pairs of 1024 tokens, d = 256: 29.5 and 33.8; backward 103.3 and 108.9); more units keep the tensor cores
    // busier in the streaming kernel.
    if (D.l_a % T != 0 || n_qt > 8) return false;
    return pairs <= resident_clusters(n_qt);
}

uoe_status launch_smha_fused(const Dims& D, const SmhaFused& f, const PlanPtrs& P, const int* patch_idx, const int* expert_idx,
                             const int* offsets, bool causal, const Rope& rope, int* status, cudaStream_t s) {
    const int n_qt = (D.l_a + T - 1) / T;
    const long long pairs = (long long)D.B * D.k;
    FuMaps tm;
    {                     // x as [B m patches, l_p rows, d]
        const uint64_t dims[3] = {(uint64_t)D.d, (uint64_t)D.l_p, (uint64_t)D.B * D.m};
        const uint64_t str[2] = {(uint64_t)D.d * 2, (uint64_t)D.d * 2 * D.l_p};
        const uint32_t box[3] = {BK, (uint32_t)D.l_p, 1};
        if (!make_tmap(&tm.x, f.x, 3, dims, str, box)) return UOE_ERR_CUDA;
    }
    for (int q = 0; q < 3; ++q) {       // W [n, d, 64] as [n][one column block][d][64]
        const uint64_t dims[4] = {64, (uint64_t)D.d, 1, (uint64_t)D.n};
        const uint64_t str[3] = {128, 128, (uint64_t)D.d * 128};
        const uint32_t box[4] = {64, BK, 1, 1};
        if (!make_tmap(&tm.w[q], f.W[q], 4, dims, str, box)) return UOE_ERR_CUDA;
    }
    tm.k = tm.v = tm.wo = tm.z = tm.x;
    if (n_qt > 1) {
        const uint64_t dims[2] = {DH, (uint64_t)D.Rmax};
        const uint64_t str[1] = {DH * 2};
        const uint32_t box[2] = {DH, T};
        if (!make_tmap(&tm.k, f.k, 2, dims, str, box) || !make_tmap(&tm.v, f.v, 2, dims, str, box)) return UOE_ERR_CUDA;
    }
    if (!f.q) {
        const uint64_t dims[3] = {(uint64_t)D.d, DH, (uint64_t)D.n};
        const uint64_t str[2] = {(uint64_t)D.d * 2, (uint64_t)D.d * DH * 2};
        const uint32_t box[3] = {64, DH, 1};
        if (!make_tmap(&tm.wo, f.Wo, 3, dims, str, box)) return UOE_ERR_CUDA;
        if (n_qt > 1) {
            const uint64_t zdims[2] = {(uint64_t)D.d, (uint64_t)D.Rmax};
            const uint64_t zstr[1] = {(uint64_t)D.d * 2};
            const uint32_t zbox[2] = {64, 32};
            if (!make_tmap(&tm.z, f.z, 2, zdims, zstr, zbox)) return UOE_ERR_CUDA;
        }
    }
    FuArgs a;
    a.q = (__nv_bfloat16*)f.q; a.k = (__nv_bfloat16*)f.k; a.v = (__nv_bfloat16*)f.v; a.o = (__nv_bfloat16*)f.o; a.z = (__nv_bfloat16*)f.z;
    a.lse = f.lse;
    a.pair_row = P.pair_row; a.patch_idx = patch_idx; a.expert_idx = expert_idx; a.expert_end = P.expert_end; a.offsets = offsets;
    a.pairs = (int)pairs; a.n = D.n; a.m = D.m; a.k_sel = D.k; a.c = D.c; a.Lv = D.Lv; a.l_a = D.l_a; a.d = D.d; a.causal = causal ? 1 : 0;
    a.n_qt = n_qt;
    a.lp_log = 0;
    while ((1 << a.lp_log) < D.l_p) ++a.lp_log;
    a.scale_log2 = 1.4426950408889634f / sqrtf((float)D.d_h);
    a.status = status;
    ProfScope ps("smha_fused", s);
    auto go = [&](auto multi, auto rot) -> uoe_status {
        constexpr bool MULTI = decltype(multi)::value, ROPE = decltype(rot)::value;
        using L = FuLaunch<MULTI, ROPE>;
        const uoe_status st = L::opt_in();
        if (st != UOE_OK) return st;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[2];
        cfg.gridDim = dim3((unsigned)(pairs * n_qt));
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = FCfg<MULTI>::SMEM;
        cfg.stream = s;
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        at[1].id = cudaLaunchAttributeClusterDimension;
        at[1].val.clusterDim.x = (unsigned)n_qt; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = MULTI ? 2 : 1;
        typename std::conditional<ROPE, Rope, NoRopeF>::type r;
        if constexpr (ROPE) r = rope;
        return cudaLaunchKernelEx(&cfg, L::kernel(), tm, a, r) == cudaSuccess ? UOE_OK : UOE_ERR_CUDA;
    };
    const bool rot = rope.pair0 < 32;
    uoe_status st;
    if (n_qt > 1) st = rot ? go(std::true_type{}, std::true_type{}) : go(std::true_type{}, std::false_type{});
    else st = rot ? go(std::false_type{}, std::true_type{}) : go(std::false_type{}, std::false_type{});
    if (st != UOE_OK) return st;
    UOE_LAUNCHED();
    return UOE_OK;
}

}  // namespace uoe
