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
// plan: grid B, 128 threads (512 when the backward asks for long per-row arrays), dynamic shared memory 8*k*c bytes.  Everything a sample needs from global memory
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
    const int b = blockIdx.x, tid = threadIdx.x, NT = blockDim.x;      // NT: 128 or 512 (long per-row arrays)
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
        for (int i = 0; i < n; ++i) {
            for (int rb = s_end[i] / l_p + tid; rb < offs[i + 1] / l_p; rb += NT) src_patch[rb] = -1;
            if (row_gate)          // padding rows weigh nothing
                for (int r = s_end[i] + tid; r < offs[i + 1]; r += NT) { row_gate[r] = 0.f; row_valid[r] = 0.f; }
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
// combine: grid (B*m, row groups)
// ---------------------------------------------------------------------------------------------
template <typename T, bool BWD /* the backward's combine: rvec and sum */>
__global__ void __launch_bounds__(kThreads)
combine_kernel(const T* __restrict__ x, const T* __restrict__ z, const int* __restrict__ inv_row,
               const float* __restrict__ inv_gate, T* __restrict__ y, int L, int Lv, int d, int m, int k,
               int l_p, int residual, int use_gate, int rows_per_cta, const float* __restrict__ rvec,
               const int* __restrict__ pair_row /* not null: inv_row holds offsets from the pair's first row */,
               const float* __restrict__ gate_bkc /* not null: whole samples per expert (slot u is patch u): no inverse map,
                                                     weights from the router's gate array [B,k,c] */, int c,
               int patches, const DwrSum sum /* total > 0: the CTAs past the patches add up dW_r (backward) */) {
    pdl_trigger();
    pdl_wait();
    if (BWD && blockIdx.x >= patches) {
        dwr_sum(sum, (int)((blockIdx.x - patches) * gridDim.y + blockIdx.y));
        return;
    }
    constexpr int V = Vec16<T>::N;
    __shared__ int srow[32];
    __shared__ float sg[32];
    const int bj = blockIdx.x, b = bj / m, j = bj % m;
    const int r0 = blockIdx.y * rows_per_cta, r1 = min(l_p, r0 + rows_per_cta);
    if (threadIdx.x < k) {
        if (gate_bkc) {          // Eq. 26: the token's row in every chosen expert follows from its position alone
            srow[threadIdx.x] = j * l_p < Lv ? pair_row[(size_t)b * k + threadIdx.x] + j * l_p : -1;
            sg[threadIdx.x] = use_gate ? gate_bkc[((size_t)b * k + threadIdx.x) * c + j] : 1.0f;
        } else {
            const int rel = inv_row[(size_t)bj * k + threadIdx.x];
            const int base = pair_row ? pair_row[(size_t)b * k + threadIdx.x] : 0;
            srow[threadIdx.x] = rel >= 0 ? rel + base : -1;
            sg[threadIdx.x] = use_gate ? inv_gate[(size_t)bj * k + threadIdx.x] : 1.0f;
        }
    }
    __syncthreads();
    const int vpr = d / V;
    const int total = (r1 - r0) * vpr;
    for (int idx = threadIdx.x; idx < total; idx += kThreads) {
        const int r = r0 + idx / vpr, cv = idx % vpr;
        const int t = j * l_p + r;
        const size_t xo = ((size_t)b * L + t) * d + (size_t)cv * V;
        // the loads of a round (x and up to four slots) are issued together, then added in ascending slot order
        const bool real = t < Lv;
        uint4 xv = make_uint4(0, 0, 0, 0), q[4];
        if (residual) xv = ld_stream16(x + xo);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (real && u < k && srow[u] >= 0) q[u] = ld_stream16(z + ((size_t)(srow[u] + r)) * d + (size_t)cv * V);
        float acc[V];
        unpack16<T>(xv, acc);
        if (real) {
            for (int s0 = 0; s0 < k; s0 += 4) {
                if (s0 > 0) {
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (s0 + u < k && srow[s0 + u] >= 0)
                            q[u] = ld_stream16(z + ((size_t)(srow[s0 + u] + r)) * d + (size_t)cv * V);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (s0 + u < k && srow[s0 + u] >= 0) {
                        float f[V];
                        unpack16<T>(q[u], f);
                        const float g = sg[s0 + u];
#pragma unroll
                        for (int v = 0; v < V; ++v) acc[v] = fmaf(g, f[v], acc[v]);
                    }
                }
            }
            if (rvec) {         // (a run-time check in the forward too: without it the compiler orders the loop above worse, d = 2432,
                                // sixteen experts, 22k tokens 176 us instead of 166)
                const float* rp = rvec + (size_t)bj * d + (size_t)cv * V;
#pragma unroll
                for (int v = 0; v < V; v += 4) {
                    const float4 rq = *(const float4*)(rp + v);
                    acc[v] += rq.x; acc[v + 1] += rq.y; acc[v + 2] += rq.z; acc[v + 3] += rq.w;
                }
            }
        }
        st_stream16(y + xo, pack16<T>(acc));
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
    const int threads = (P.row_gate && (long long)D.k * D.l_a >= 4096) ? 512 : 128;      // the backward's per-row weights: k*l_a rows per sample
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
    // 16-byte vectors per thread: two for small outputs (short dependent chains, many CTAs in flight: these launches are
    // bound by latency), four to eight once the output is tens of MB (fewer, longer CTAs: less set-up per byte; measured
    // 35 -> 31 us at 44 MB, 198 -> 183 us at 268 MB)
    const long long out_bytes = (long long)D.B * D.L * D.d * D.esize;
    const int vecs = out_bytes < (32ll << 20) ? 2 : (out_bytes < (128ll << 20) ? 4 : 8);
    int rows_per_cta = (int)(vecs * kThreads * 16 / ((long long)D.d * D.esize));
    if (rows_per_cta < 1) rows_per_cta = 1;
    if (rows_per_cta > D.l_p) rows_per_cta = D.l_p;
    // the additions of dW_r take whole columns of the grid (one row of it for them, the rest of the columns idle, was 84 us
    // instead of 19 at d = 1408, n = 24 with ten patches of 64 tokens: 46000 empty CTAs)
    const int row_groups = (D.l_p + rows_per_cta - 1) / rows_per_cta;
    dim3 grid(D.B * D.m + (dwr_sum_blocks(sum) + row_groups - 1) / row_groups, row_groups);
    const bool ident = P.inv_relative && P.identity_patches && P.gate != nullptr;
    const long long ctas = (long long)grid.x * grid.y;
    ProfScope ps("combine", s);
    auto go = [&](SpreadOnce& once, auto kern, auto elem) {
        using T = decltype(elem);
        launch_k(kern, grid, dim3(kThreads), spread_smem(once, kern, ctas, 0), s, (const T*)x, (const T*)z, (const int*)P.inv_row,
                 (const float*)P.inv_gate, (T*)y, D.L, D.Lv, D.d, D.m, D.k, D.l_p, residual ? 1 : 0, use_gate ? 1 : 0, rows_per_cta,
                 rvec, P.inv_relative ? (const int*)P.pair_row : (const int*)nullptr, ident ? P.gate : (const float*)nullptr, D.c,
                 D.B * D.m, sum);
    };
    static SpreadOnce once[3];
    if (!D.bf16) go(once[0], combine_kernel<float, false>, float());
    else if (rvec || sum.total > 0) go(once[1], combine_kernel<__nv_bfloat16, true>, __nv_bfloat16());
    else go(once[2], combine_kernel<__nv_bfloat16, false>, __nv_bfloat16());
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
