// Weight gradients of a whole backward half in one launch, for matrices too small to give every SM several 256 x 256
// tiles (those go to wgrad_tcgen05.cu):   dW[e] [M, N] = P_e^T Q_e  for up to two problems (UoME: dW1 and dW2; SMHA: the
// three projections side by side, and the output projection), P_e, Q_e the rows of expert e's region.
//
// The contraction runs over the ragged row count of each expert, so both operands are "MN-major" for the MMA: a K step is
// consecutive rows, each row contributing 128 bytes (64 elements) per swizzled column block.  Either operand may be
// gathered from the source tensor (Eq. 18 inside the contraction): a 64-row K block is then 64 / l_p slabs of l_p rows,
// one copy each with all the column blocks of the tile, laid out [slab][column block][l_p rows][128 bytes]; the MMA's
// descriptors carry the slab's strides, so 16-row patches cost four copies per operand and K block, not four per column
// block.
//
// Work split: an output tile is 128 x BN (BN <= 256); its cost is its 64-row K blocks times the time of one, of which more
// than two thirds are the same for every width (kStepCost).  The tiles of both problems form one line (wgrad_line.h), cut
// into equal pieces, one per CTA (one CTA per SM; fewer where the line is too short for that), whatever the load of the experts.
// A tile inside one piece is written straight to its output; a tile cut by pieces leaves one partial tile per piece in
// the scratch, and wgrad_reduce adds them in ascending order (in spare CTAs of router_grad_kernel, or as a
// launch of its own).  No CTA waits for another, every sum has a fixed order.
//   warp 0      TMA producer, four-stage ring (P block [64 x 128], Q block [64 x BN])
//   warp 1      MMA issuer: tcgen05.mma 128 x BN x 16, two accumulator sets (the write-out of a tile runs under the next)
//   warps 2-9   write-out, two per TMEM lane quarter, 32-column chunks in turn
#include "kernels.cuh"
#include "launch_rules.h"
#include "tc.cuh"
#include "tmap.cuh"
#include "wgrad_stream.cuh"

namespace uoe {
namespace {

using namespace tc;

constexpr int BM = kLineBM, BK = kLineBK, BN_MAX = kLineBNMax;
constexpr int P_BYTES = BM * BK * 2, Q_BYTES = BN_MAX * BK * 2, STAGE = P_BYTES + Q_BYTES;
constexpr int STAGES = 4;
constexpr int EPI_WARPS = 8, THREADS = 64 + 32 * EPI_WARPS, STG_BYTES = 32 * 128;
constexpr int CTL_BYTES = 2048;
constexpr int SMEM = STAGES * STAGE + 1024 /*align slack*/ + CTL_BYTES + EPI_WARPS * STG_BYTES;

struct SCtl {
    uint64_t full[STAGES], empty[STAGES], tfull[2], tempty[2];
    uint32_t tmem_base;
    int abort_flag;
    int offs[34];
    WSched sched;
};
static_assert(sizeof(SCtl) <= CTL_BYTES, "control block");

struct WMaps { CUtensorMap P, Q, out[3]; };     // out: [n*M, out_cols] float32 in [32 x 32] pieces (not used when transposed)
struct WOperand { int gather, nslab, sub; };    // a K block is nslab slabs of sub rows
struct WArgs {
    WProblem prob[2];
    WOperand p[2], q[2];
    WMaps maps[2];
    const int* offsets;
    const int* src_patch;
    float* part;
    int* status;
    int n, nprob, l_p, Bm, pieces, part_floats;
};

__global__ void __launch_bounds__(THREADS, 1)
wgrad_stream_kernel(const __grid_constant__ WArgs a) {
    pdl_trigger();
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    SCtl* ctl = (SCtl*)(smem + STAGES * STAGE);
    volatile int* abort_flag = &ctl->abort_flag;
    int* status = a.status;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 1); }
        for (int q = 0; q < 2; ++q) { mbar_init(&ctl->tfull[q], 1); mbar_init(&ctl->tempty[q], 32 * EPI_WARPS); }
        ctl->abort_flag = 0;
        fence_barrier_init();
        for (int p = 0; p < a.nprob; ++p) { prefetch_tmap(&a.maps[p].P); prefetch_tmap(&a.maps[p].Q); }
    }
    if (warp == 1) tmem_alloc(&ctl->tmem_base, 512);
    pdl_wait();                     // everything above touches only this CTA's own resources
    if (warp == 2) {
        const int o = a.offsets[min(lane, a.n)];
        ctl->offs[lane] = o;
        if (lane == 0) ctl->offs[a.n] = a.offsets[a.n];
        __syncwarp();
        wsched_build(ctl->sched, ctl->offs, a.n, a.prob, a.nprob, a.pieces, lane);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    const WSched& sc = ctl->sched;
    const int c = blockIdx.x;

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        int stage = 0;
        uint32_t phase = 0, issued = 0, issued_parity = 0;
        bool stop = false;
        const int lp_shift = __ffs(a.l_p) - 1;               // gathered operands: l_p is a power of two that divides 128
        WFrag f;
        for (int pos = c * sc.Q; !stop && wsched_next(sc, a.prob, c, pos, f);) {
            if (f.kb_lo >= f.kb_hi) continue;
            const WProblem& pr = a.prob[f.p];
            const WMaps& tm = a.maps[f.p];
            const WOperand &op = a.p[f.p], &oq = a.q[f.p];
            const uint32_t bytes = P_BYTES + pr.BN * BK * 2;
            const bool gathers = op.gather || oq.gather;
            // lanes 0-15 serve P, 16-31 Q: lane (slab) issues its own copy
            const WOperand& mine = lane < 16 ? op : oq;
            const int slab = lane & 15;
            const bool active = slab < (mine.gather ? mine.nslab : 1);
            const int blk0 = lane < 16 ? f.m0 / 64 : f.n0 / 64, nblk = lane < 16 ? BM / 64 : pr.BN / 64;
            const CUtensorMap* map = lane < 16 ? &tm.P : &tm.Q;
            const uint32_t dst0 = (lane < 16 ? 0 : P_BYTES) + (mine.gather ? slab * mine.sub * 128 * nblk : 0);
            // Source patches of the gathered rows: the warp keeps 32 consecutive entries of src_patch in its lanes and
            // reads them with a shuffle (a look-up in global memory in front of every copy would set the ring's pace)
            const int r0 = ctl->offs[f.e] + f.kb_lo * BK;
            const int patch_end = gathers ? (r0 + (f.kb_hi - f.kb_lo) * BK + a.l_p - 1) >> lp_shift : 0;
            int win0 = r0 >> lp_shift;
            int win = (gathers && win0 + lane < patch_end) ? a.src_patch[win0 + lane] : 0;
            for (int kb = f.kb_lo; kb < f.kb_hi; ++kb) {
                const int row = r0 + (kb - f.kb_lo) * BK;
                int src = 0, prow = 0;
                if (gathers) {
                    if (((row + BK - 1) >> lp_shift) >= win0 + 32) {      // (uniform) the block's last slab is past the window
                        win0 = row >> lp_shift;
                        win = win0 + lane < patch_end ? a.src_patch[win0 + lane] : 0;
                    }
                    const int srow = row + (mine.gather ? slab * mine.sub : 0);
                    src = __shfl_sync(0xffffffffu, win, ((srow >> lp_shift) - win0) & 31);
                    if (src < 0) src = a.Bm;                              // no patch: the zero-filled box past the end
                    prow = srow & (a.l_p - 1);
                }
                int ok = 1;
                if (lane == 0) ok = (mbar_wait(&ctl->empty[stage], phase ^ 1, abort_flag, status) && !*abort_flag) ? 1 : 0;
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) { stop = true; break; }
                uint8_t* dst = smem + stage * STAGE + dst0;
                if (lane == 0) mbar_arrive_expect_tx(&ctl->full[stage], bytes);
                __syncwarp();
                if (active) {
                    if (mine.gather) tma_load_4d(dst, map, 0, prow, blk0, src, &ctl->full[stage]);
                    else tma_load_3d(dst, map, 0, row, blk0, &ctl->full[stage]);
                }
                issued |= 1u << stage;
                issued_parity = (issued_parity & ~(1u << stage)) | (phase << stage);
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
        }
        if (lane == 0 && *abort_flag) {      // let this CTA's own copies land before it exits
            for (int s = 0; s < STAGES; ++s)
                if (issued & (1u << s)) mbar_wait(&ctl->full[s], (issued_parity >> s) & 1, abort_flag, status);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (the whole warp, one elected lane issues) ----------------
        const uint32_t el = elect_one();
        int stage = 0, acc = 0;
        uint32_t phase = 0, acc_phase = 0;
        bool stop = false;
        WFrag f;
        for (int pos = c * sc.Q; !stop && wsched_next(sc, a.prob, c, pos, f);) {
            const WProblem& pr = a.prob[f.p];
            const WOperand &op = a.p[f.p], &oq = a.q[f.p];
            const uint32_t idesc = instr_desc_bf16(BM, f.cols, true, true);
            // strides of a K-block's slabs: rows of a slab are consecutive, column blocks a slab's size apart; with
            // eight-row slabs the second eight rows of a K step lie in the next slab
            const int subp = op.gather ? op.sub : BK, subq = oq.gather ? oq.sub : BK, nbq = pr.BN / 64;
            const uint32_t lbo_p = subp * 128, sbo_p = subp == 8 ? 2048 : 1024;
            const uint32_t lbo_q = subq * 128, sbo_q = subq == 8 ? nbq * 1024 : 1024;
            uint32_t po[BK / 16], qo[BK / 16];
#pragma unroll
            for (int ks = 0; ks < BK / 16; ++ks) {
                po[ks] = (16 * ks / subp) * (subp * 256) + (16 * ks % subp) * 128;
                qo[ks] = (16 * ks / subq) * (subq * 128 * nbq) + (16 * ks % subq) * 128;
            }
            if (!mbar_wait_warp(&ctl->tempty[acc], acc_phase ^ 1, abort_flag, status)) break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + acc * BN_MAX;
            for (int kb = f.kb_lo; kb < f.kb_hi; ++kb) {
                if (!mbar_wait_warp(&ctl->full[stage], phase, abort_flag, status)) { stop = true; break; }
                tc_fence_after();
                const uint32_t sp = smem_u32(smem + stage * STAGE), sq = sp + P_BYTES;
#pragma unroll
                for (int ks = 0; ks < BK / 16; ++ks)
                    mma_bf16(el, d_tmem, smem_desc(sp + po[ks], lbo_p, sbo_p), smem_desc(sq + qo[ks], lbo_q, sbo_q), idesc,
                             kb > f.kb_lo || ks > 0);
                mma_commit(el, &ctl->empty[stage]);
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
            if (stop) break;
            mma_commit(el, &ctl->tfull[acc]);
            if (++acc == 2) { acc = 0; acc_phase ^= 1; }
        }
    } else {
        // ---------------- write-out ----------------
        const int quarter = warp & 3, wsel = (warp - 2) >> 2;
        uint8_t* stg = smem + STAGES * STAGE + CTL_BYTES + (warp - 2) * STG_BYTES;
        int acc = 0;
        uint32_t acc_phase = 0;
        WFrag f;
        for (int pos = c * sc.Q; wsched_next(sc, a.prob, c, pos, f);) {
            const WProblem& pr = a.prob[f.p];
            const bool ready = mbar_wait(&ctl->tfull[acc], acc_phase, abort_flag, status) && !*abort_flag;
            if (!__all_sync(0xffffffffu, ready)) break;      // warp-uniform: tcgen05.ld below is warp-collective
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN_MAX;
            const int row = quarter * 32 + lane;
            float4* part = (float4*)(a.part + wsched_slot(f, c) * (size_t)a.part_floats);
#pragma unroll 1
            for (int ch = wsel; ch < f.cols / 32; ch += 2) {
                uint32_t v[32];
                if (f.kb_lo < f.kb_hi) {
                    tmem_ld32(taddr + ch * 32, v);
                    tmem_ld_wait();
                } else {
#pragma unroll
                    for (int q = 0; q < 32; ++q) v[q] = 0u;
                }
                if (f.c_first != f.c_last) {         // a partial tile: [column / 4][row] of four floats, whole lines per store
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        part[(ch * 8 + q) * BM + row] = make_float4(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]),
                                                                    __uint_as_float(v[4 * q + 2]), __uint_as_float(v[4 * q + 3]));
                } else if (pr.transposed) {          // out [n, N, M]: a column of the tile is 128 consecutive floats
                    float* o = pr.out[0] + ((size_t)f.e * pr.N + f.n0 + ch * 32) * pr.M + f.m0 + row;
#pragma unroll
                    for (int q = 0; q < 32; ++q) o[(size_t)q * pr.M] = __uint_as_float(v[q]);
                } else {
                    const int col = f.n0 + ch * 32, which = col / pr.out_cols;
                    if (lane == 0) bulk_wait_read();      // the previous store has finished reading the piece
                    __syncwarp();
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        *(uint4*)(stg + lane * 128 + ((q ^ (lane & 7)) << 4)) = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_2d(&a.maps[f.p].out[which], stg, col - which * pr.out_cols, f.e * pr.M + f.m0 + quarter * 32);
                        bulk_commit();
                    }
                }
            }
            tc_fence_before();
            mbar_arrive(&ctl->tempty[acc]);
            if (++acc == 2) { acc = 0; acc_phase ^= 1; }
        }
    }
    if (warp >= 2 && lane == 0) bulk_wait_all();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tmem_dealloc(tmem_base, 512);
    }
}

__global__ void __launch_bounds__(kReduceThreads)
wgrad_reduce_kernel(const __grid_constant__ WReduce r) {
    pdl_trigger();
    pdl_wait();
    wgrad_reduce(r, blockIdx.x);
}

}  // namespace

size_t wgrad_stream_scratch_bytes(const int (*mn)[2], int nprob, int n, long long rows_max) {
    WTileShape t[2];
    for (int i = 0; i < nprob; ++i) t[i] = wgrad_tile_shape(mn[i][0], mn[i][1]);
    return (size_t)wgrad_scratch_floats(t, nprob, n, rows_max) * sizeof(float);
}

uoe_status launch_wgrad_stream(const WStreamProblem* probs, int nprob, const int* offsets, int n, long long rows_max,
                               const int* src_patch, int l_p, int Bm, float* part, const char* label, int* status, cudaStream_t s,
                               WReduce* reduce) {
    if (nprob < 1 || nprob > 2 || n > 32 || !part) return UOE_ERR_UNSUPPORTED;
    static DeviceOnce once;
    {
        const uoe_status st = smem_opt_in(once, wgrad_stream_kernel, SMEM);
        if (st != UOE_OK) return st;
    }
    WArgs a;
    a.offsets = offsets; a.src_patch = src_patch; a.part = part; a.status = status;
    a.n = n; a.nprob = nprob; a.l_p = l_p > 0 ? l_p : 64; a.Bm = Bm;
    WTileShape shape[2];
    int wmax = 0, widest = 0;
    for (int i = 0; i < nprob; ++i) {
        const WStreamProblem& in = probs[i];
        if (in.M % BM != 0 || in.N % 64 != 0) return UOE_ERR_UNSUPPORTED;
        if ((in.gather_p || in.gather_q) && (!src_patch || l_p < 8 || 128 % l_p != 0)) return UOE_ERR_INVALID_ARG;
        WProblem& p = a.prob[i];
        p.M = in.M; p.N = in.N; p.transposed = in.transposed ? 1 : 0;
        p.out_cols = in.out_cols > 0 ? in.out_cols : in.N;
        for (int q = 0; q < 3; ++q) p.out[q] = in.out[q];
        const WTileShape t = shape[i] = wgrad_tile_shape(in.M, in.N);
        p.BN = t.BN; p.m_tiles = t.m_tiles; p.n_tiles = t.n_tiles; p.w = t.w;
        if (t.w > wmax) wmax = t.w;
        if (t.BN > widest) widest = t.BN;
        const int sub = l_p < BK ? l_p : BK;
        auto operand = [&](WOperand& o, CUtensorMap* tm, const void* base, int cols, int nblk, bool gather) {
            o.gather = gather ? 1 : 0; o.sub = gather ? sub : BK; o.nslab = BK / o.sub;
            if (gather) {      // [Bm patches][column blocks][l_p rows][64]
                const uint64_t dims[4] = {64, (uint64_t)l_p, (uint64_t)cols / 64, (uint64_t)Bm};
                const uint64_t str[3] = {(uint64_t)cols * 2, 128, (uint64_t)cols * 2 * l_p};
                const uint32_t box[4] = {64, (uint32_t)sub, (uint32_t)nblk, 1};
                return make_tmap(tm, base, 4, dims, str, box);
            }
            const uint64_t dims[3] = {64, (uint64_t)rows_max, (uint64_t)cols / 64};
            const uint64_t str[2] = {(uint64_t)cols * 2, 128};
            const uint32_t box[3] = {64, BK, (uint32_t)nblk};
            return make_tmap(tm, base, 3, dims, str, box);
        };
        if (!operand(a.p[i], &a.maps[i].P, in.P, in.M, BM / 64, in.gather_p) ||
            !operand(a.q[i], &a.maps[i].Q, in.Q, in.N, p.BN / 64, in.gather_q))
            return UOE_ERR_CUDA;
        for (int q = 0; q < 3; ++q) {
            const uint64_t dims[2] = {(uint64_t)p.out_cols, (uint64_t)n * p.M};
            const uint64_t str[1] = {(uint64_t)p.out_cols * 4};
            const uint32_t box[2] = {32, 32};
            float* o = in.out[q] ? in.out[q] : in.out[0];
            if (p.transposed) a.maps[i].out[q] = a.maps[i].P;
            else if (!make_tmap(&a.maps[i].out[q], o, 2, dims, str, box, CU_TENSOR_MAP_DATA_TYPE_FLOAT32)) return UOE_ERR_CUDA;
        }
    }
    const long long bound = wgrad_line_bound(shape, nprob, n, rows_max);
    a.pieces = wgrad_pieces(bound, wmax, sm_count());
    a.part_floats = (int)wgrad_part_floats(widest);
    if (!wgrad_line_fits(bound, wmax, a.pieces)) return UOE_ERR_UNSUPPORTED;
    {
        ProfScope ps(label, s);
        launch_k(wgrad_stream_kernel, dim3(a.pieces), dim3(THREADS), (size_t)SMEM, s, a);
    }
    UOE_LAUNCHED();
    WReduce r;
    r.prob[0] = a.prob[0];
    r.prob[1] = a.prob[nprob - 1];
    r.offsets = offsets; r.part = part; r.n = n; r.nprob = nprob; r.pieces = a.pieces;
    r.part_floats = a.part_floats;
    int tiles = 0;
    for (int i = 0; i < nprob; ++i) tiles += n * a.prob[i].m_tiles * a.prob[i].n_tiles;
    r.by_cut = tiles > a.pieces - 1 ? 1 : 0;
    r.halves = widest / 32 * 8;
    r.places = r.by_cut ? a.pieces - 1 : tiles;
    r.use_threads(router_grad_threads(r.by_cut != 0, 0, 0));
    *reduce = r;
    return UOE_OK;
}

uoe_status launch_wgrad_reduce(const WReduce& r, cudaStream_t s) {
    if (r.blocks == 0) return UOE_OK;
    ProfScope ps("wgrad_reduce", s);
    static SpreadOnce once;
    launch_k(wgrad_reduce_kernel, dim3(r.blocks), dim3(r.threads), spread_smem(once, wgrad_reduce_kernel, r.blocks, 0), s, r);
    UOE_LAUNCHED();
    return UOE_OK;
}

}  // namespace uoe
