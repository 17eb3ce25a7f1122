// Data movement around the expert GEMMs: the routing plan, the token gather (Eq. 18 / 24), the
// weighted combine (Eq. 20 / 26 / 40), and the float32 grouped GEMM used by the float32 path.
#include "kernels.cuh"

namespace uoe {
namespace {

constexpr int kThreads = 256;

// ---------------------------------------------------------------------------------------------
// pair rows for many samples: one CTA passes over expert_idx [B,k] once, a warp per expert, 32 samples per step,
// and writes where every (sample, slot) pair's rows start (samples, then slots ascending inside an expert's region) and
// the table that leads back from there.  O(B k) work in all, where plan_kernel's own scan of the earlier samples is
// O(B k) per sample.
// ---------------------------------------------------------------------------------------------
constexpr int kPlanScanMaxB = 512;        // up to here every sample's CTA scans the earlier samples itself

__global__ void __launch_bounds__(1024)
plan_rows_kernel(const int* __restrict__ expert_idx, const int* __restrict__ offsets, int B, int n, int k, int l_a,
                 int* __restrict__ pair_row, int* __restrict__ slot_pair, int slot_shift) {
    pdl_trigger();
    pdl_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = warp; i < n; i += 32) {
        const int off_i = offsets[i];
        int running = 0;
        for (int b0 = 0; b0 < B; b0 += 32) {
            const int b = b0 + lane;
            unsigned slots = 0;                 // this sample's slots that name expert i (a caller's routing may repeat one)
            if (b < B)
                for (int s = 0; s < k; ++s)
                    if (expert_idx[(size_t)b * k + s] == i) slots |= 1u << s;
            const unsigned ball = __ballot_sync(0xffffffffu, slots != 0u);
            int q = running + __popc(ball & ((1u << lane) - 1u));
            running += __popc(ball);
            if (__any_sync(0xffffffffu, slots & (slots - 1u))) {      // more than one slot of a sample: count slots, not samples
                int incl = __popc(slots);
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += v;
                }
                q = running - __popc(ball) + incl - __popc(slots);
                running += __shfl_sync(0xffffffffu, incl, 31) - __popc(ball);
            }
            for (unsigned left = slots; left; left &= left - 1, ++q) {
                const int pair = b * k + __ffs(left) - 1;
                pair_row[pair] = off_i + q * l_a;
                slot_pair[pair_slot_by_row(off_i, q, slot_shift)] = pair;
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------
// plan: grid B, 128 threads (512 when the backward asks for per-row arrays), dynamic shared memory 8*k*c bytes.  Everything a sample needs from global memory
// (its routing arrays, the offsets, the expert choices of the samples before it) is fetched in one round of
// independent loads; the rest runs out of shared memory.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(512)
plan_kernel(const int* __restrict__ expert_idx, const int* __restrict__ patch_idx, const float* __restrict__ gate,
            const int* __restrict__ offsets, int B, int n, int k, int m, int c, int l_p,
            int* __restrict__ pair_row, int* __restrict__ inv_row, float* __restrict__ inv_gate,
            int* __restrict__ expert_end, int* status, float* __restrict__ row_gate, float* __restrict__ row_valid,
            int Lv, int use_gate, int* __restrict__ src_patch, const PlanTails tails,
            long long rows_max, int rows_given /* pair_row and slot_pair are already there (plan_rows_kernel) */,
            int* __restrict__ slot_pair, int slot_shift) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ int s_dyn[];
    int* s_pi = s_dyn;                         // [k*c] patch indices of this sample
    float* s_g = (float*)(s_dyn + k * c);      // [k*c] gates
    // A slot that names no expert is reported and given the last rows that hold a pair, so that whatever goes by pairs stays
    // inside the buffers (its sample's results mean nothing; no other sample reads those rows).
    __shared__ int my_e[32], prow[32], hist[33], offs[34];
    const int b = blockIdx.x, tid = threadIdx.x, NT = blockDim.x;      // NT: 128 or 512 (per-row arrays)
    const int l_a = c * l_p;
    if (tid < 33) hist[tid] = 0;
    __syncthreads();
    // ---- one round of loads ----
    if (tid < k) {
        int e = expert_idx[b * k + tid];
        if (e < 0 || e >= n) { set_status(status, UOE_ERR_DEVICE_INDEX); e = -1; }
        my_e[tid] = e;
    }
    if (tid <= n) offs[tid] = offsets[tid];
    for (int idx = tid; idx < k * c; idx += NT) {
        const int pj = patch_idx[(size_t)b * k * c + idx];
        if (pj < -1 || pj >= m) set_status(status, UOE_ERR_DEVICE_INDEX);
        s_pi[idx] = pj;
        s_g[idx] = gate[(size_t)b * k * c + idx];
    }
    if (!rows_given) {   // choices of the samples before b, per expert: lane i of each warp counts expert i through ballots
        int acc = 0;
        const int lane = tid & 31;
        for (int i0 = 0; i0 < b * k; i0 += NT) {
            const int idx = i0 + tid;
            const int e = idx < b * k ? expert_idx[idx] : -1;
            for (int i = 0; i < n; ++i) {
                const unsigned msk = __ballot_sync(0xffffffffu, e == i);
                if (lane == i) acc += __popc(msk);
            }
        }
        if (lane < n && acc) atomicAdd(&hist[lane], acc);
    }
    __syncthreads();
    if (tid < k) {
        const int e = my_e[tid];
        // pairs of this expert in front of this one: of earlier samples, and of this one (a caller's routing may repeat an expert)
        const unsigned same = __match_any_sync(k < 32 ? (1u << k) - 1u : 0xffffffffu, e);
        int row = (int)rows_max - l_a;
        if (e >= 0) {
            const int q = hist[e] + __popc(same & ((1u << tid) - 1u));
            row = rows_given ? pair_row[b * k + tid] : offs[e] + q * l_a;
            if (!rows_given) slot_pair[pair_slot_by_row(offs[e], q, slot_shift)] = b * k + tid;
        }
        prow[tid] = row;
        if (!rows_given || e < 0) pair_row[b * k + tid] = row;
    }
    __syncthreads();
    for (int idx = tid; idx < m * k; idx += NT) {          // inverse map: which routed rows feed patch j
        const int j = idx / k, s = idx % k;
        int slot = -1;
        for (int u = 0; u < c; ++u)
            if (s_pi[s * c + u] == j) slot = u;
        inv_row[((size_t)b * m + j) * k + s] = slot >= 0 ? prow[s] + slot * l_p : -1;
        inv_gate[((size_t)b * m + j) * k + s] = slot >= 0 ? s_g[s * c + slot] : 0.f;
    }
    // source patch of every l_p-row block (used when the GEMM gathers its own A operand)
    for (int idx = tid; idx < k * c; idx += NT) {
        const int s = idx / c, u = idx % c;
        const int pj = s_pi[idx];
        src_patch[prow[s] / l_p + u] = (pj >= 0 && pj < m) ? b * m + pj : -1;
    }
    if (b == B - 1) {          // the last sample has seen every choice: ends of the expert regions, padding blocks
        __shared__ int s_end[32];
        if (rows_given) {      // the last pair of a region starts l_a rows before its end: the largest first row per expert
            if (tid < n) s_end[tid] = offs[tid];
            __syncthreads();
            for (int idx = tid; idx < B * k; idx += NT) {
                const int e = expert_idx[idx];
                if (e >= 0 && e < n) atomicMax(&s_end[e], pair_row[idx] + l_a);
            }
            __syncthreads();
            if (tid < n) expert_end[tid] = s_end[tid];
        } else {
            if (tid < k && my_e[tid] >= 0) atomicAdd(&hist[my_e[tid]], 1);
            __syncthreads();
            if (tid < n) s_end[tid] = expert_end[tid] = offs[tid] + hist[tid] * l_a;
        }
        __syncthreads();
        for (int i = tid >> 5; i < n; i += NT >> 5) {          // a warp per expert
            for (int rb = s_end[i] / l_p + (tid & 31); rb < offs[i + 1] / l_p; rb += 32) src_patch[rb] = -1;
            if (row_gate)          // padding rows weigh nothing
                for (int r = s_end[i] + (tid & 31); r < offs[i + 1]; r += 32) { row_gate[r] = 0.f; row_valid[r] = 0.f; }
        }
    }
    if (tails.row_bytes > 0) {
        const long long r0 = offs[n], row_vecs = tails.row_bytes / 16;
        const long long total = (min(rows_max, r0 + 128) - r0) * row_vecs;
        for (long long q = (long long)b * NT + tid; q < total; q += (long long)B * NT)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (tails.p[i]) ((uint4*)tails.p[i])[r0 * row_vecs + q] = make_uint4(0, 0, 0, 0);
    }
    if (row_gate) {                          // per-row weights for the backward
        for (int idx = tid; idx < k * l_a; idx += NT) {
            const int s = idx / l_a, r = idx % l_a, u = r / l_p;
            const int pj = s_pi[s * c + u];
            const bool real = pj >= 0 && pj < m && pj * l_p + (r % l_p) < Lv;
            const float g = use_gate ? s_g[s * c + u] : 1.0f;
            row_gate[prow[s] + r] = real ? g : 0.f;
            row_valid[prow[s] + r] = real ? 1.f : 0.f;
        }
    }
}

// ---------------------------------------------------------------------------------------------
// gather: grid (B*k*c + n, nsplit); a patch is one contiguous slab of l_p*d elements on both sides
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads)
gather_kernel(const uint4* __restrict__ src, const int* __restrict__ patch_idx, const int* __restrict__ offsets,
              const int* __restrict__ pair_row, const int* __restrict__ expert_end,
              uint4* __restrict__ dst, int n_slabs, int k, int c, int m, long long slab_vecs /* l_p*d*esize/16 */,
              long long row_vecs /* d*esize/16 */, int l_p, int n, uint4* __restrict__ tail, long long tail_row_vecs,
              long long rows_max) {
    pdl_trigger();
    pdl_wait();
    const int bx = blockIdx.x;
    long long count;                 // 16-byte pieces to write
    const uint4* s = nullptr;
    uint4* o;
    if (bx == n_slabs + n) {         // rows of `tail` that no kernel writes
        const long long r0 = offsets[n];
        o = tail + r0 * tail_row_vecs;
        count = (rows_max - r0) * tail_row_vecs;
    } else if (bx < n_slabs) {
        const int pair = bx / c, u = bx % c, b = pair / k;
        const int j = patch_idx[bx];
        o = dst + ((long long)pair_row[pair] + (long long)u * l_p) * row_vecs;
        count = slab_vecs;
        if (j >= 0 && j < m) s = src + ((long long)b * m + j) * slab_vecs;
    } else {
        const int i = bx - n_slabs;
        const long long r0 = expert_end[i], r1 = offsets[i + 1];
        o = dst + r0 * row_vecs;
        count = (r1 - r0) * row_vecs;
    }
    const long long per = (count + gridDim.y - 1) / gridDim.y;
    const long long lo = per * blockIdx.y, hi = min(count, lo + per);
    if (s) {
        long long i = lo + threadIdx.x;
        for (; i + 3 * kThreads < hi; i += 4 * kThreads) {
            uint4 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = ld_stream16(s + i + q * kThreads);
#pragma unroll
            for (int q = 0; q < 4; ++q) st_stream16(o + i + q * kThreads, v[q]);
        }
        for (; i < hi; i += kThreads) st_stream16(o + i, ld_stream16(s + i));
    } else {
        const uint4 z = make_uint4(0, 0, 0, 0);
        for (long long i = lo + threadIdx.x; i < hi; i += kThreads) st_stream16(o + i, z);
    }
}

// ---------------------------------------------------------------------------------------------
// combine: a patch is one contiguous slab of x, of y and of every routed buffer that holds it, so y is a weighted sum of
// slabs.  Bound by memory: the warps of a persistent grid work for themselves on units of 2 x 32 16-byte vectors of a slab,
// the next unit's rows and weights (a lane per slot), this unit's x and its first two slots in flight together, and no
// step waits for another warp.  (A CTA per 4 to 16 KB of output, which looks its slots up, meets, and then loads: thousands
// of short CTAs, 7.2 us against 6.5 at 8 MB of output, 13 and 10 at 17 MB, 29 and 24 at 44 MB = 6.4 TB/s; image block forward
// 220.5 -> 211, its training step 715 -> 704, long-document block 91.3 -> 85.4.  One vector per lane: 225 us, the four: 216 for
// the image block; three or four slots in flight: 216 and 217.  With up to sixteen slots per patch, two / four in flight: 16 samples of 1024
// tokens, d = 512, 495.6 / 499.5 us, 4 of them 165.5 / 171.2; one sample 87.0 / 82.9, d = 256 74.3 / 72.3, where the rounds are a chain.)
// ---------------------------------------------------------------------------------------------
constexpr int kCombineVecs = 2, kCombineSlots = 2;

struct CombineArgs {
    const void *x, *z;
    void* y;
    const int* inv_row;
    const float* inv_gate;
    const int* pair_row;        // not null: inv_row holds offsets from the pair's first row
    const float* gate_bkc;      // not null: whole samples per expert (slot u is patch u): no inverse map, weights from the
                                // router's gate array [B,k,c]
    const float* rvec;
    int Lv, m, k, c, l_p, vpr /* vectors per row */, chunks /* units per slab */, units, residual, use_gate;
    DwrSum sum;                 // backward: added up behind the units, from the last warp on (the last have the fewest units)
};

template <typename T, bool BWD /* the backward's combine: rvec and sum */>
__global__ void __launch_bounds__(kThreads)
combine_kernel(const CombineArgs a) {
    pdl_trigger();
    pdl_wait();
    constexpr int V = Vec16<T>::N, U = kCombineVecs, S = kCombineSlots;
    const int lane = threadIdx.x & 31, warps = (int)gridDim.x * (kThreads / 32);
    int unit = (int)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5);
    // slot `lane` of a patch: its first routed row (-1: none) and weight
    auto look_up = [&](int bj, int& row, float& g) {
        row = -1;
        g = 1.0f;
        if (lane >= a.k) return;
        const int b = bj / a.m, j = bj - b * a.m;
        if (a.gate_bkc) {            // Eq. 26: the token's row in every chosen expert follows from its position alone
            if (j * a.l_p < a.Lv) row = a.pair_row[(size_t)b * a.k + lane] + j * a.l_p;
            if (a.use_gate) g = j < a.c ? a.gate_bkc[((size_t)b * a.k + lane) * a.c + j] : 0.f;
        } else {
            const int rel = a.inv_row[(size_t)bj * a.k + lane];
            const int base = a.pair_row ? a.pair_row[(size_t)b * a.k + lane] : 0;
            if (rel >= 0) row = rel + base;
            if (a.use_gate) g = a.inv_gate[(size_t)bj * a.k + lane];
        }
    };
    int bj = unit / a.chunks, row_next = -1;
    float g_next = 0.f;
    if (unit < a.units) look_up(bj, row_next, g_next);
    while (unit < a.units) {
        const int v0 = (unit - bj * a.chunks) * (32 * U) + lane;             // this lane's first vector of the slab
        const int j = bj % a.m, slab = a.l_p * a.vpr, real = max(0, min(a.l_p, a.Lv - j * a.l_p)) * a.vpr;
        const size_t at = (size_t)bj * slab;
        const int row = row_next;
        const float g = g_next;
        uint4 xv[U], q[S][U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            xv[u] = make_uint4(0, 0, 0, 0);
            if (a.residual && v0 + 32 * u < slab) xv[u] = ld_stream16((const uint4*)a.x + at + v0 + 32 * u);
        }
        unsigned slots = __ballot_sync(0xffffffffu, row >= 0);              // the patch's routed copies, taken in ascending order
        unsigned held = slots;                                              // those whose vectors are on their way or here
        auto load = [&]() {                                                 // the next S of them
#pragma unroll
            for (int i = 0; i < S; ++i) {
                if (!slots) break;
                const uint4* zp = (const uint4*)a.z + (size_t)__shfl_sync(0xffffffffu, row, __ffs(slots) - 1) * a.vpr;
                slots &= slots - 1;
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (v0 + 32 * u < real) q[i][u] = ld_stream16(zp + v0 + 32 * u);
            }
        };
        load();
        unit += warps;
        const int bj_this = bj;
        bj = unit / a.chunks;
        if (unit < a.units) look_up(bj, row_next, g_next);
        float acc[U][V];
#pragma unroll
        for (int u = 0; u < U; ++u) unpack16<T>(xv[u], acc[u]);
        while (held) {
#pragma unroll
            for (int i = 0; i < S; ++i) {
                if (!held) break;
                const float w = __shfl_sync(0xffffffffu, g, __ffs(held) - 1);
                held &= held - 1;
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (v0 + 32 * u < real) {
                        float f[V];
                        unpack16<T>(q[i][u], f);
#pragma unroll
                        for (int v = 0; v < V; ++v) acc[u][v] = fmaf(w, f[v], acc[u][v]);
                    }
            }
            if (held) load();
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int v = v0 + 32 * u;
            if (BWD && a.rvec && v < real) {
                const float* rp = a.rvec + ((size_t)bj_this * a.vpr + v % a.vpr) * V;
#pragma unroll
                for (int w = 0; w < V; w += 4) {
                    const float4 rq = *(const float4*)(rp + w);
                    acc[u][w] += rq.x; acc[u][w + 1] += rq.y; acc[u][w + 2] += rq.z; acc[u][w + 3] += rq.w;
                }
            }
            if (v < slab) st_stream16((uint4*)a.y + at + v, pack16<T>(acc[u]));
        }
    }
    if (BWD) {
        const int items = (a.sum.total + kDwrItem - 1) / kDwrItem;
        for (int i = warps - 1 - ((int)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)); i < items; i += warps) dwr_sum(a.sum, i);
    }
}

// ---------------------------------------------------------------------------------------------
// float32 grouped GEMM on the FFMA pipes: TM x TN tile, MT x NT outputs per thread, KG groups of threads that share
// the tile and take the BK-deep K steps' columns in turn (their sums are added in group order at the end).  A three-stage
// cp.async ring; A is kept [row][k] and read four k at a time, its rows dealt round robin to the threads so that the
// reads of a warp hit different banks.  A may be gathered: single rows of x, any patch length (Eq. 18).
// Two shapes.  Large problems: 128 x 64, 8 x 8 per thread (FFMA-bound: 16 multiply-adds per 16-byte shared-memory read).
// Small ones, where the chain of K steps and idle SMs are the bound: 32 x 32 with four K groups (256 x 256 matrices over
// 512 rows: 128 CTAs, each thread 64 of the 256 k's).
// ---------------------------------------------------------------------------------------------
template <int TM, int TN, int MT, int NT, int KG, int BK> struct F32Cfg {
    static constexpr int GROUP = (TM / MT) * (TN / NT);          // threads of a K group
    static constexpr int THREADS = GROUP * KG;
    static constexpr int LDA = BK + 4;                           // floats per A row: adjacent rows start four banks apart
    static constexpr int STAGE = TM * LDA + BK * TN;             // floats
    static constexpr int STAGES = 3;
    static constexpr int RED = KG > 1 ? (KG - 1) * TM * TN : 0;
    static constexpr int SMEM = (STAGES * STAGE > RED ? STAGES * STAGE : RED) * 4 + TM * 8;
    static_assert(STAGE % 2 == 0 && RED % 2 == 0, "the row indices behind the ring are 8-byte aligned");
    static_assert(128 % TM == 0 && BK % (4 * KG) == 0 && NT % 4 == 0, "tile shape");
};

template <int TM, int TN, int MT, int NT, int KG, int BK>
__global__ void __launch_bounds__(F32Cfg<TM, TN, MT, NT, KG, BK>::THREADS)
gemm_f32_kernel(const float* __restrict__ A, const float* __restrict__ W, const float* __restrict__ bias,
                float* __restrict__ C, float* __restrict__ pre, const int* __restrict__ offsets, int n, int K, int N,
                int act, int gathered, const SrcMap map) {
    using Cf = F32Cfg<TM, TN, MT, NT, KG, BK>;
    pdl_trigger();
    pdl_wait();
    extern __shared__ __align__(16) float s_ring[];
    long long* s_src = (long long*)(s_ring + (Cf::SMEM - TM * 8) / 4);       // source row of every tile row, -1 = zeros
    const int row0 = blockIdx.x * TM, col0 = blockIdx.y * TN, tid = threadIdx.x;
    if (row0 >= offsets[n]) return;
    int e = 0;
    while (e + 1 < n && row0 >= offsets[e + 1]) ++e;             // regions are multiples of 128 rows: no tile straddles
    for (int r = tid; r < TM; r += Cf::THREADS) s_src[r] = gathered ? source_row(map, row0 + r, e, offsets[e]) : row0 + r;
    __syncthreads();
    const float* We = W + (size_t)e * K * N;
    const int steps = (K + BK - 1) / BK;

    auto copy = [](float* dst, const float* src, bool valid) {   // 16 bytes, zero-filled when not valid
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                     :: "r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(valid ? 16 : 0) : "memory");
    };
    auto load = [&](int step) {
        if (step < steps) {
            float* sa = s_ring + (step % Cf::STAGES) * Cf::STAGE;
            float* sb = sa + TM * Cf::LDA;
            const int k0 = step * BK;
            for (int q = tid; q < TM * BK / 4; q += Cf::THREADS) {
                const int r = q / (BK / 4), kk = (q % (BK / 4)) * 4;
                const long long src = s_src[r];
                const bool ok = src >= 0 && k0 + kk < K;
                copy(sa + r * Cf::LDA + kk, ok ? A + (size_t)src * K + k0 + kk : A, ok);
            }
            for (int q = tid; q < BK * TN / 4; q += Cf::THREADS) {
                const int kk = q / (TN / 4), cc = (q % (TN / 4)) * 4;
                const bool ok = k0 + kk < K && col0 + cc < N;
                copy(sb + kk * TN + cc, ok ? We + (size_t)(k0 + kk) * N + col0 + cc : We, ok);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int st = 0; st < Cf::STAGES - 1; ++st) load(st);

    const int g = tid / Cf::GROUP, t = tid % Cf::GROUP;
    constexpr int TX = TN / NT, TY = TM / MT;
    const int tx = t % TX, ty = t / TX;
    float acc[MT][NT] = {};
    for (int step = 0; step < steps; ++step) {
        asm volatile("cp.async.wait_group %0;" :: "n"(Cf::STAGES - 2) : "memory");
        __syncthreads();                      // this step has landed for every thread, and the step before it has been read
        load(step + Cf::STAGES - 1);
        const float* sa = s_ring + (step % Cf::STAGES) * Cf::STAGE;
        const float* sb = sa + TM * Cf::LDA;
#pragma unroll
        for (int q = 0; q < BK / (4 * KG); ++q) {
            const int kk = (q * KG + g) * 4;
            float4 a[MT];
#pragma unroll
            for (int i = 0; i < MT; ++i) a[i] = *(const float4*)(sa + (i * TY + ty) * Cf::LDA + kk);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float b[NT];
#pragma unroll
                for (int j = 0; j < NT / 4; ++j) {
                    const float4 v = *(const float4*)(sb + (kk + u) * TN + j * (TN / (NT / 4)) + tx * 4);
                    b[4 * j] = v.x; b[4 * j + 1] = v.y; b[4 * j + 2] = v.z; b[4 * j + 3] = v.w;
                }
#pragma unroll
                for (int i = 0; i < MT; ++i) {
                    const float av = u == 0 ? a[i].x : (u == 1 ? a[i].y : (u == 2 ? a[i].z : a[i].w));
#pragma unroll
                    for (int j = 0; j < NT; ++j) acc[i][j] = fmaf(av, b[j], acc[i][j]);
                }
            }
        }
    }
    if (KG > 1) {                             // add the K groups' sums in group order
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if (g > 0) {
#pragma unroll
            for (int i = 0; i < MT; ++i)
#pragma unroll
                for (int j = 0; j < NT; ++j) s_ring[((g - 1) * MT * NT + i * NT + j) * Cf::GROUP + t] = acc[i][j];
        }
        __syncthreads();
        if (g > 0) return;
#pragma unroll
        for (int q = 0; q < KG - 1; ++q)
#pragma unroll
            for (int i = 0; i < MT; ++i)
#pragma unroll
                for (int j = 0; j < NT; ++j) acc[i][j] += s_ring[(q * MT * NT + i * NT + j) * Cf::GROUP + t];
    }
#pragma unroll
    for (int j = 0; j < NT / 4; ++j) {
        const int cc = col0 + j * (TN / (NT / 4)) + tx * 4;
        if (cc >= N) continue;                // N is a multiple of four
        float4 bv = make_float4(0.f, 0.f, 0.f, 0.f);
        if (bias) bv = *(const float4*)(bias + (size_t)e * N + cc);
#pragma unroll
        for (int i = 0; i < MT; ++i) {
            const size_t o = (size_t)(row0 + i * TY + ty) * N + cc;
            float4 v = make_float4(acc[i][4 * j] + bv.x, acc[i][4 * j + 1] + bv.y, acc[i][4 * j + 2] + bv.z, acc[i][4 * j + 3] + bv.w);
            if (pre) *(float4*)(pre + o) = v;
            v.x = act_apply(v.x, act); v.y = act_apply(v.y, act); v.z = act_apply(v.z, act); v.w = act_apply(v.w, act);
            *(float4*)(C + o) = v;
        }
    }
}

// 128 x 64 tiles from here on (a little over one per SM); below, 32 x 32 tiles.  Whole forward, us with the large / small tiles
// (256 x 256 experts): 76 tiles 71 / 47, 140 tiles 70 / 64;  512 x 384 experts, 400 tiles 218 / 246, 800 tiles 390 / 475.
// (64 x 64 tiles with scalar copies, the only shape before: 177, 165, 414, 703.)
constexpr long long kF32LargeTiles = 160;

}  // namespace

uoe_status launch_plan(const Dims& D, const int* expert_idx, const int* patch_idx, const float* gate,
                       const int* offsets, const PlanPtrs& P, int* status, cudaStream_t s, bool use_gate, const PlanTails& tails) {
    const size_t smem = (size_t)D.k * D.c * 8;
    if (smem > 32 * 1024) return UOE_ERR_UNSUPPORTED;      // a sample's routing arrays live in shared memory
    const bool many = D.B > kPlanScanMaxB;
    if (many) {
        ProfScope ps("plan_rows", s);
        launch_k(plan_rows_kernel, dim3(1), dim3(1024), 0, s, expert_idx, offsets, D.B, D.n, D.k, D.l_a, P.pair_row, P.slot_pair,
                 pair_slot_shift(D.l_a));
        UOE_LAUNCHED();
    }
    ProfScope ps("plan", s);
    const int threads = P.row_gate ? 512 : 128;      // the backward's per-row weights: k*l_a rows per sample (image block, training step: 672 us with 128, 670 so)
    launch_k(plan_kernel, dim3(D.B), dim3(threads), smem, s, expert_idx, patch_idx, gate, offsets, D.B, D.n, D.k, D.m, D.c, D.l_p,
                                    P.pair_row, P.inv_row, P.inv_gate, P.expert_end, status, P.row_gate, P.row_valid,
                                    D.Lv, use_gate ? 1 : 0, P.src_patch, tails, D.Rmax, many ? 1 : 0, P.slot_pair, pair_slot_shift(D.l_a));
    UOE_LAUNCHED();
    return UOE_OK;
}

uoe_status launch_gather(const Dims& D, const void* src, const int* patch_idx, const int* offsets,
                         const PlanPtrs& P, void* dst, cudaStream_t s, void* tail, long long tail_row_bytes) {
    const long long row_vecs = (long long)D.d * D.esize / 16;
    const long long slab_vecs = row_vecs * D.l_p;
    const int n_slabs = D.B * D.k * D.c;
    int nsplit = (int)((slab_vecs * 16 + 16383) / 16384);
    if (nsplit < 1) nsplit = 1;
    if (nsplit > 128) nsplit = 128;
    dim3 grid(n_slabs + D.n + (tail ? 1 : 0), nsplit);
    static SpreadOnce once;
    ProfScope ps("gather", s);
    launch_k(gather_kernel, grid, dim3(kThreads), spread_smem(once, gather_kernel, (long long)grid.x * grid.y, 0), s, (const uint4*)src, patch_idx, offsets, P.pair_row, P.expert_end,
                                            (uint4*)dst, n_slabs, D.k, D.c, D.m, slab_vecs, row_vecs, D.l_p, D.n,
                                            (uint4*)tail, tail_row_bytes / 16, D.Rmax);
    UOE_LAUNCHED();
    return UOE_OK;
}

uoe_status launch_combine(const Dims& D, const void* x, const void* z, const PlanPtrs& P, bool residual,
                          bool use_gate, void* y, cudaStream_t s, const float* rvec, const DwrSum& sum) {
    const int vpr = (int)((long long)D.d * D.esize / 16);
    const long long chunks = ((long long)D.l_p * vpr + 32 * kCombineVecs - 1) / (32 * kCombineVecs), units = (long long)D.B * D.m * chunks;
    if ((long long)D.l_p * vpr > (1ll << 31) - 16384 || units > (1ll << 31) - 16384) return UOE_ERR_UNSUPPORTED;      // the kernel counts both in 32 bits
    CombineArgs a;
    a.x = x; a.z = z; a.y = y; a.inv_row = P.inv_row; a.inv_gate = P.inv_gate;
    a.pair_row = P.inv_relative ? P.pair_row : nullptr;
    a.gate_bkc = P.inv_relative && P.identity_patches ? P.gate : nullptr;
    a.rvec = rvec;
    a.Lv = D.Lv; a.m = D.m; a.k = D.k; a.c = D.c; a.l_p = D.l_p; a.vpr = vpr;
    a.residual = residual ? 1 : 0; a.use_gate = use_gate ? 1 : 0;
    a.sum = sum;
    ProfScope ps("combine", s);
    const bool bwd = rvec || sum.total > 0;
    a.chunks = (int)chunks;
    a.units = (int)units;
    // Four CTAs per SM, all that fit (up to eight) only for a forward with several units per warp even then: the room is of
    // use to the next kernel, whose CTAs start under this one (language-model training step 257 us with four, 262 with eight;
    // wide block forward 167.5 and 165.4)
    const int per_sm = !bwd && a.units >= 10 * (kThreads / 32) * sm_count() ? 8 : 4;
    const int want = (a.units + kThreads / 32 - 1) / (kThreads / 32), cap = per_sm * sm_count();
    const dim3 grid(want < cap ? want : cap);
    // A unit per warp: CTAs kept apart (block forwards, without and with: 304 CTAs 76.8 and 69.5 us, 112 CTAs 76.7 and 72.4, 498 CTAs 65.2
    // and 61.8).  Not where warps go on to further units, there the room is the next kernel's (training steps, 592 CTAs: 172.4 and 173.9,
    // 251.2 and 253.5).
    auto go = [&](SpreadOnce& once, auto kern) {
        launch_k(kern, grid, dim3(kThreads), want < cap ? spread_smem(once, kern, grid.x, 0) : 0, s, a);
    };
    static SpreadOnce once[3];
    if (!D.bf16) go(once[0], combine_kernel<float, false>);
    else if (bwd) go(once[1], combine_kernel<__nv_bfloat16, true>);
    else go(once[2], combine_kernel<__nv_bfloat16, false>);
    UOE_LAUNCHED();
    return UOE_OK;
}

uoe_status launch_gemm_f32(const GemmArgs& g, cudaStream_t s) {
    if (g.b_kmajor || g.nmat != 1 || (g.K & 3) || (g.N & 3)) return UOE_ERR_UNSUPPORTED;
    ProfScope ps(g.label, s);
    auto go = [&](SpreadOnce& once, auto kern, int tm, int tn, int threads, int smem) {
        const uoe_status st = smem_opt_in(once.opt_in, kern, 160 * 1024);
        if (st != UOE_OK) return st;
        const dim3 grid((unsigned)((g.rows_max + tm - 1) / tm), (g.N + tn - 1) / tn);
        launch_k(kern, grid, dim3(threads), spread_smem(once, kern, (long long)grid.x * grid.y, (size_t)smem), s,
                 (const float*)(g.gather_x ? g.gather_x : g.A), (const float*)g.W, (const float*)g.bias, (float*)g.C, (float*)g.pre,
                 g.offsets, g.n, g.K, g.N, g.act, g.gather_x ? 1 : 0, g.map);
        return UOE_OK;
    };
    using Large = F32Cfg<128, 64, 8, 8, 1, 16>;
    using Small = F32Cfg<32, 32, 4, 4, 4, 32>;
    static SpreadOnce once[2];
    const long long large_tiles = g.rows_max / 128 * ((g.N + 63) / 64);
    const uoe_status st = large_tiles >= kF32LargeTiles
                              ? go(once[0], gemm_f32_kernel<128, 64, 8, 8, 1, 16>, 128, 64, Large::THREADS, Large::SMEM)
                              : go(once[1], gemm_f32_kernel<32, 32, 4, 4, 4, 32>, 32, 32, Small::THREADS, Small::SMEM);
    if (st != UOE_OK) return st;
    UOE_LAUNCHED();
    return UOE_OK;
}

}  // namespace uoe
