// uoe_mlp_backward: gradients of sum(y * dy) for y = uoe_mlp_forward(x, ...) with the selection held
// constant (derivative of Eq. 38-40; with gating also of Eq. 14 and 21 through the gate weights).
//
// In routed-row space, for a row r of expert i with combine weight w_r, saved pre-activation h_r:
//   u_r  = dy_r A^O_i^T                      grouped GEMM (K-major weights), epilogue produces
//   dh_r = w_r u_r * phi'(h_r)               -> buffer dh
//   ag_r = w_r phi(h_r)                      -> buffer ag
//   dgate(slab) = sum_r <u_r, phi(h_r)>      -> per-row partials, reduced per (sample, expert, patch)
//   dA^O_i = ag^T dy_g,  dA^I_i = x_g^T dh   ragged-K weight-gradient GEMMs
//   dx_g = dh A^I_i^T                        grouped GEMM, then combined back with unit weights
// Router: dgate -> dP_samp, dP_patch -> softmax Jacobians -> per-(sample, patch) logit gradient G, which
// feeds dW_r (through the pooled token sums) and one more term of dx.
#include "balance.cuh"
#include "kernels.cuh"
#include "launch_rules.h"
#include "tc.cuh"
#include "tmap.cuh"

namespace uoe {
namespace {

using namespace tc;

// Gradient of the router logits of one sample from the per-row gate gradients.  grid B, 256 or 512 threads, dynamic shared
// memory (2 n m + k c) floats.  A warp per slab adds the slab's per-row, per-column-tile partials (fixed order), then the
// softmax Jacobians of Eq. 14 and 21:  G[b,j,i] = dlogit_patch[b,i,j]/cnt_j + dlogit_samp[b,i]/L_valid.
// Latency-bound (a sample's partials are a few KB to a few hundred KB); one launch instead of a slab-sum kernel and a
// Jacobian kernel whose sums over a slot list were one thread's serial loop.
__global__ void __launch_bounds__(kReduceThreads, 2)
router_grad_kernel(const float* __restrict__ dg_part, int nt, const int* __restrict__ pair_row,
                   const int* __restrict__ expert_idx, const int* __restrict__ patch_idx,
                   const float* __restrict__ p_samp, const float* __restrict__ p_patch, int n, int k, int m, int c,
                   int l_p, int Lv, float* __restrict__ G, int B,
                   const __grid_constant__ WReduce reduce /* reduce.blocks further CTAs add up cut weight-gradient tiles */) {
    pdl_trigger();
    pdl_wait();
    // the samples first where they are few (their slab sums are long chains), last where they would hold the additions up
    const int b = B <= 64 ? (int)blockIdx.x : (int)blockIdx.x - reduce.blocks;
    if (b < 0 || b >= B) {
        wgrad_reduce(reduce, b < 0 ? (int)blockIdx.x : b - B);
        return;
    }
    extern __shared__ float sm[];
    float* pp = sm;                 // [n][m] patch gate
    float* dpp = sm + n * m;        // [n][m] its gradient
    float* dg = sm + 2 * n * m;     // [k][c] gradient of the combine weight of every slot
    __shared__ float ps[32], dls[32], dps[32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, NT = blockDim.x;
    for (int idx = tid; idx < n * m; idx += NT) { pp[idx] = p_patch[(size_t)b * n * m + idx]; dpp[idx] = 0.f; }
    if (tid < 32) { ps[tid] = tid < n ? p_samp[(size_t)b * n + tid] : 0.f; dps[tid] = 0.f; }
    // four slabs at a time, so that their look-ups and loads are in flight together (one at a time a sample of 1271 slabs of
    // four tokens took 90 us)
    const int len = l_p * nt;
    constexpr int U = 4;
    for (int slab0 = warp * U; slab0 < k * c; slab0 += NT / 32 * U) {
        const float* src[U];
        int n_q[U];                                       // values of the slab: none of an unused slot
        float a[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int slab = min(slab0 + u, k * c - 1);
            const int j = patch_idx[(size_t)b * k * c + slab];
            src[u] = dg_part + ((size_t)pair_row[b * k + slab / c] + (size_t)(slab % c) * l_p) * nt;
            n_q[u] = j >= 0 && j < m ? len : 0;
            a[u] = 0.f;
        }
        int q = lane;
        for (; q + 96 < len; q += 128) {
            float t[U][4];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int w = 0; w < 4; ++w) t[u][w] = n_q[u] ? src[u][q + 32 * w] : 0.f;
#pragma unroll
            for (int u = 0; u < U; ++u) a[u] += (t[u][0] + t[u][1]) + (t[u][2] + t[u][3]);
        }
        for (; q < len; q += 32) {
#pragma unroll
            for (int u = 0; u < U; ++u) a[u] += n_q[u] ? src[u][q] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a[u] += __shfl_xor_sync(0xffffffffu, a[u], o);
            if (lane == 0 && slab0 + u < k * c) dg[slab0 + u] = a[u];
        }
    }
    __syncthreads();
    // gate = P_samp * P_patch: a warp per chosen expert, lanes over its slots
    for (int s = warp; s < k; s += NT / 32) {
        int i = expert_idx[(size_t)b * k + s];
        i = (unsigned)i < (unsigned)n ? i : 0;            // (the plan kernel has reported an index out of range)
        float acc = 0.f;
        for (int u = lane; u < c; u += 32) {
            const int j = patch_idx[((size_t)b * k + s) * c + u];
            if (j < 0 || j >= m) continue;
            acc += dg[s * c + u] * pp[i * m + j];
            dpp[i * m + j] = dg[s * c + u] * ps[i];      // one (expert, patch) pair per slot: no other writer
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) dps[i] = acc;
    }
    __syncthreads();
    if (warp == 0) {                                      // softmax Jacobian of the sample gate (Eq. 21)
        float dot = ps[lane] * dps[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
        dls[lane] = ps[lane] * (dps[lane] - dot);
    }
    __syncthreads();
    for (int j = tid; j < m; j += NT) {         // softmax Jacobian of each patch gate (Eq. 14)
        const int cnt = max(0, min(l_p, Lv - j * l_p));
        float dot = 0.f;
        for (int i = 0; i < n; ++i) dot += pp[i * m + j] * dpp[i * m + j];
        for (int i = 0; i < n; ++i) {
            const float dlp = pp[i * m + j] * (dpp[i * m + j] - dot);
            G[((size_t)b * m + j) * n + i] = cnt > 0 ? dlp / (float)cnt + dls[i] / (float)Lv : 0.f;
        }
    }
}

// What the router's logit gradient G [B*m, n] does to W_r and x, in one pass over x:
//   dW_r[dd, i] = sum over (b, j) of pool[bj, dd] G[bj, i],  pool = sum of the real rows of patch bj
//   rvec[bj, dd] = sum_i W_r[dd, i] G[bj, i], which every real token of the patch receives in dx
// Bound by reading x once.  Grid (blocks of 64 columns, splits of the patches), two CTAs per SM in all.  Every warp streams
// for itself: it takes each eighth patch of its CTA's range through its own ring of TMA stages (at most 32 rows of 64
// columns each), a lane adds two columns up over the rows and multiplies them, so no step waits for another warp and
// the pooled tensor never reaches memory.  At the end the warps' dW_r meet in shared memory; every split leaves its own
// partial (dwr_sum adds them in split order).  SPREAD: the vector is written to every row of dx at once instead of to
// rvec (the balance loss, whose whole dx it is).
// Against CTA-wide batches (16-byte loads a batch ahead in registers, sums through shared memory, two to four CTA barriers
// per batch: a chain of barriers and 750 instructions per warp and batch, the same through TMA stages), us, cold caches:
// B = 256, L = 224, d = 384, n = 6: 20.8 -> 17.0;  B = 16, L = 512, d = 512, n = 8: 8.8 -> 6.7;  B = 4, L = 2048, d = 1024,
// n = 8: 10.5 -> 8.2;  B = 8, L = 4096, d = 4096, n = 16: 70 -> 48 (5.5 TB/s);  SPREAD, B = 16, L = 2048, d = 1024,
// n = 16: 34 -> 24.4.  (A pooling kernel, product kernels and a vector or spreading kernel before that: 58, 22, -, 77, 84.)
constexpr int kApplyWarps = 8, kApplyCols = 64, kApplyRows = 32, kApplyStages = 8, kApplyRing = 3 * kApplyRows * kApplyCols * 2;
struct ApplyArgs {
    const __nv_bfloat16* W_r;
    const float* G;
    float *rvec, *part;
    __nv_bfloat16* dx;
    int* status;
    int patches, Lv, d, n, m, l_p, nseg, seg_rows, per, stages;
};
template <int NMAX, bool SPREAD>
__global__ void __launch_bounds__(32 * kApplyWarps, NMAX > 16 ? 1 : 2)
router_apply_kernel(const __grid_constant__ CUtensorMap xmap /* x as [B m, l_p, d], boxes of [seg_rows, 64] */, const ApplyArgs a) {
    pdl_trigger();
    extern __shared__ uint8_t s_raw[];
    __shared__ uint64_t full[kApplyWarps][kApplyStages];
    __shared__ int s_abort;
    __shared__ __align__(16) float2 sG[kApplyWarps][NMAX];              // (g, g)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n = a.n, d = a.d, nseg = a.nseg, unit_bytes = a.seg_rows * kApplyCols * 2;
    uint8_t* smem = (uint8_t*)(((uintptr_t)s_raw + 127) & ~(uintptr_t)127);
    uint8_t* ring = smem + warp * a.stages * unit_bytes;
    volatile int* abort_flag = &s_abort;
    if (tid == 0) s_abort = 0;
    if (lane == 0) {
        for (int s = 0; s < a.stages; ++s) mbar_init(&full[warp][s], 1);
        fence_barrier_init();
        prefetch_tmap(&xmap);
    }
    __syncthreads();
    const int c0 = blockIdx.x * kApplyCols, dd = c0 + 2 * lane;       // this lane's columns: dd and dd + 1 (d is a multiple of eight)
    const int first = blockIdx.y * a.per + warp, end = min(a.patches, (int)(blockIdx.y + 1) * a.per);
    int ip = first, is = 0, st_in = 0;                // the next copy: patch, segment, stage
    auto issue = [&]() {
        if (ip >= end) return;
        if (lane == 0) {
            mbar_arrive_expect_tx(&full[warp][st_in], (uint32_t)unit_bytes);
            tma_load_3d(ring + st_in * unit_bytes, &xmap, c0, is * a.seg_rows, ip, &full[warp][st_in]);
        }
        if (++st_in == a.stages) st_in = 0;
        if (++is == nseg) { is = 0; ip += kApplyWarps; }
    };
    pdl_wait();
    for (int s = 0; s < a.stages; ++s) issue();
    float g_next = first < end && lane < n ? a.G[(size_t)first * n + lane] : 0.f;
    unsigned long long acc[NMAX], w[NMAX];            // pairs over the two columns
#pragma unroll
    for (int i = 0; i < NMAX; ++i) {
        const bool in = i < n && dd < d;
        acc[i] = 0ull;
        w[i] = in ? f2_pack(__bfloat162float(a.W_r[(size_t)dd * n + i]), __bfloat162float(a.W_r[(size_t)(dd + 1) * n + i])) : 0ull;
    }
    int st = 0;                                       // the stage that is read next
    uint32_t phase = 0;
    bool ok = true;
    for (int patch = first; ok && patch < end; patch += kApplyWarps) {
        const int j = patch % a.m, real = max(0, min(a.l_p, a.Lv - j * a.l_p));
        unsigned long long p = 0ull;
        for (int seg = 0; seg < nseg; ++seg) {
            ok = mbar_wait_warp(&full[warp][st], phase, abort_flag, a.status);
            if (!ok) break;
            const int rows = min(a.seg_rows, real - seg * a.seg_rows);
            const uint8_t* src = ring + st * unit_bytes + lane * 4;
            auto add = [&](uint32_t t) { f2_add(p, f2_pack(__uint_as_float(t << 16), __uint_as_float(t & 0xffff0000u))); };
            int r = 0;
            for (; r + 7 < rows; r += 8) {
                uint32_t t[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) t[u] = *(const uint32_t*)(src + (r + u) * (kApplyCols * 2));
#pragma unroll
                for (int u = 0; u < 8; ++u) add(t[u]);
            }
            for (; r < rows; ++r) add(*(const uint32_t*)(src + r * (kApplyCols * 2)));
            __syncwarp();                             // the stage has been read
            issue();
            if (++st == a.stages) { st = 0; phase ^= 1; }
        }
        if (!ok) break;
        if (lane < NMAX) sG[warp][lane] = make_float2(g_next, g_next);     // zero past the experts
        __syncwarp();
        g_next = patch + kApplyWarps < end && lane < n ? a.G[(size_t)(patch + kApplyWarps) * n + lane] : 0.f;
        unsigned long long rv2 = 0ull;
#pragma unroll
        for (int i = 0; i < NMAX; i += 2) {
            const ulonglong2 g = *(const ulonglong2*)(&sG[warp][i]);
            f2_fma(acc[i], p, g.x);
            f2_fma(rv2, w[i], g.x);
            f2_fma(acc[i + 1], p, g.y);
            f2_fma(rv2, w[i + 1], g.y);
        }
        __syncwarp();
        const float2 rv = f2_unpack(rv2);
        if (!SPREAD) {
            if (dd < d) *(float2*)(a.rvec + (size_t)patch * d + dd) = rv;
        } else {                                      // four lanes' columns to one: a store covers four rows
            const __nv_bfloat162 t2 = __floats2bfloat162_rn(rv.x, rv.y);
            const uint32_t t = *(const uint32_t*)&t2;
            const int q = 4 * (lane & 7), col = c0 + 8 * (lane & 7);
            const uint4 v = make_uint4(__shfl_sync(0xffffffffu, t, q), __shfl_sync(0xffffffffu, t, q + 1),
                                       __shfl_sync(0xffffffffu, t, q + 2), __shfl_sync(0xffffffffu, t, q + 3));
            if (col < d) {
                __nv_bfloat16* o = a.dx + ((size_t)patch * a.l_p + (lane >> 3)) * d + col;
#pragma unroll 4
                for (int r = lane >> 3; r < a.l_p; r += 4, o += (size_t)4 * d) st_stream16(o, r < real ? v : make_uint4(0, 0, 0, 0));
            }
        }
    }
    if (!ok && lane == 0)                             // winding down: let this warp's own copies land before the CTA exits
        for (int s = 0; s < a.stages; ++s) {          // (stages without a copy in flight just run out of polls)
            mbar_wait(&full[warp][st], phase, abort_flag, a.status);
            if (++st == a.stages) { st = 0; phase ^= 1; }
        }
    if (!__syncthreads_and(ok)) return;               // (uniform) a copy did not arrive
    // ---- the warps' sums, ascending ----
    float* red = (float*)smem;                        // [warps][64 columns][NMAX + 1]
#pragma unroll
    for (int i = 0; i < NMAX; ++i)
        if (i < n) {
            const float2 t = f2_unpack(acc[i]);
            red[(warp * kApplyCols + 2 * lane) * (NMAX + 1) + i] = t.x;
            red[(warp * kApplyCols + 2 * lane + 1) * (NMAX + 1) + i] = t.y;
        }
    __syncthreads();
    const int outs = min(kApplyCols, d - c0) * n;
    for (int idx = tid; idx < outs; idx += 32 * kApplyWarps) {
        const int cc = idx / n, i = idx - cc * n;
        float sum = 0.f;
#pragma unroll
        for (int q = 0; q < kApplyWarps; ++q) sum += red[(q * kApplyCols + cc) * (NMAX + 1) + i];
        a.part[((size_t)blockIdx.y * d + c0) * n + idx] = sum;
    }
}

constexpr int kDwrThreads = 64;
__global__ void __launch_bounds__(kDwrThreads)
dwr_sum_kernel(const DwrSum s) {
    pdl_trigger();
    pdl_wait();
    dwr_sum(s, (int)blockIdx.x * (kDwrThreads / 32) + (threadIdx.x >> 5));
}

// Segments, stages and splits of router_apply_kernel for a problem.
struct ApplyShape { int nseg, seg_rows, stages, col_blocks, splits, per; };
ApplyShape apply_shape(const Dims& D) {
    ApplyShape a;
    a.col_blocks = (D.d + kApplyCols - 1) / kApplyCols;
    a.nseg = (D.l_p + kApplyRows - 1) / kApplyRows;
    a.seg_rows = (D.l_p + a.nseg - 1) / a.nseg;
    a.stages = kApplyRing / (a.seg_rows * kApplyCols * 2);         // 12 KB in flight per warp; less with patches of up to 11 rows,
                                                                   // whose stages are capped
    if (a.stages > kApplyStages) a.stages = kApplyStages;
    const int patches = D.B * D.m;
    // a full wave at two CTAs per SM of 148 (with more than 16 experts the kernel fits once: two waves).  Not the device's own SM
    // count: the partial sums, and with them the last bits of dW_r, follow the split, and the workspace query the shape.
    const int cap = 2 * 148 / a.col_blocks > 1 ? 2 * 148 / a.col_blocks : 1;
    a.per = (patches + cap - 1) / cap;
    a.splits = (patches + a.per - 1) / a.per;
    return a;
}
template <bool SPREAD>
uoe_status launch_router_apply(const Dims& D, const ApplyShape& a, const void* x, const void* W_r, const float* G, float* rvec,
                               float* part, void* dx, int* status, cudaStream_t s) {
    CUtensorMap xmap;
    const uint64_t dims[3] = {(uint64_t)D.d, (uint64_t)D.l_p, (uint64_t)D.B * D.m}, str[2] = {(uint64_t)D.d * 2, (uint64_t)D.d * 2 * D.l_p};
    const uint32_t box[3] = {(uint32_t)kApplyCols, (uint32_t)a.seg_rows, 1};
    if (!make_tmap(&xmap, x, 3, dims, str, box, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, CU_TENSOR_MAP_SWIZZLE_NONE)) return UOE_ERR_CUDA;
    ApplyArgs p;
    p.W_r = (const __nv_bfloat16*)W_r; p.G = G; p.rvec = rvec; p.part = part; p.dx = (__nv_bfloat16*)dx; p.status = status;
    p.patches = D.B * D.m; p.Lv = D.Lv; p.d = D.d; p.n = D.n; p.m = D.m; p.l_p = D.l_p; p.nseg = a.nseg;
    p.seg_rows = a.seg_rows; p.per = a.per; p.stages = a.stages;
    auto go = [&](SpreadOnce& once, auto kern, int nmax) {
        const uoe_status so = smem_opt_in(once.opt_in, kern, 160 * 1024);
        if (so != UOE_OK) return so;
        const size_t ring = (size_t)kApplyWarps * a.stages * a.seg_rows * kApplyCols * 2;
        const size_t red = (size_t)kApplyWarps * kApplyCols * (nmax + 1) * 4;
        launch_k(kern, dim3(a.col_blocks, a.splits), dim3(32 * kApplyWarps),
                 spread_smem(once, kern, (long long)a.col_blocks * a.splits, (ring > red ? ring : red) + 128), s, xmap, p);
        return UOE_OK;
    };
    ProfScope ps("router_apply", s);
    static SpreadOnce once[3];
    if (D.n <= 8) return go(once[0], router_apply_kernel<8, SPREAD>, 8);
    if (D.n <= 16) return go(once[1], router_apply_kernel<16, SPREAD>, 16);
    return go(once[2], router_apply_kernel<32, SPREAD>, 32);
}

// Gradient of the load-balancing loss (Eq. 42-44) with respect to the router logits.  grid B, dynamic shared memory
// n (m + 1) floats.  f_i (Eq. 43) is piecewise constant, so only P_i (Eq. 44) carries a gradient:
//   dL_b/dg_{i,j} = alpha f_i / l on the real patches;  G[b,j,i] = softmax Jacobian (Eq. 14) of that, / cnt_j.
__global__ void __launch_bounds__(kBalanceThreads)
balance_bwd_kernel(const float* __restrict__ p_patch, const float* __restrict__ dloss, int Lv, int n, int k, int m,
                   int l_p, float alpha, float* __restrict__ G) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ float s_gate[];
    __shared__ int cnts[32];
    const int b = blockIdx.x, tid = threadIdx.x;
    const int n_elig = (Lv + l_p - 1) / l_p;
    const float scale = dloss[b] * alpha * (float)n / ((float)k * (float)n_elig * (float)n_elig);     // dloss alpha (n / k l) / l
    balance_load(p_patch, b, n, m, s_gate);
    __syncthreads();
    balance_count(s_gate, n, k, m, n_elig, cnts, nullptr);
    __syncthreads();
    // scale cnts[i] is dL_b/dg of expert i; a thread per (patch, expert), in the order of G; the dot product over the experts is each thread's own
    for (int idx = tid; idx < n * m; idx += kBalanceThreads) {
        const int j = idx / n, i = idx - j * n;
        const int cnt = max(0, min(l_p, Lv - j * l_p));
        float dot = 0.f;
#pragma unroll 8
        for (int q = 0; q < n; ++q) dot += s_gate[q * (m + 1) + j] * scale * (float)cnts[q];
        const float dl = s_gate[i * (m + 1) + j] * (scale * (float)cnts[i] - dot);
        G[(size_t)b * m * n + idx] = cnt > 0 ? dl / (float)cnt : 0.f;
    }
}

struct BwdWs { size_t plan, dyg, xg, dh, ag, dxg, dgp, G, rvec, wpart, wgpart, total; int nt; };

// Which kernel takes the two weight gradients: whole tiles (wgrad_tcgen05.cu) or a line of tiles cut into equal pieces
// (wgrad_stream_tcgen05.cu).  The pieces fill the SMs whatever the number of tiles, but at any moment the CTAs work all over
// the line, so that operands larger than L2 (126 MB) are read from memory once per tile: 844 us against 574 for both gradients
// at d = 1536, d_e = 896, n = 24, 82k routed rows; 454 against 330 at d = 2048, d_e = 1024, n = 8, 32k rows, x and dy gathered.
// With fewer tiles than SMs, or operands in L2, whole tiles lose: n = 2, d = 512, d_e = 256, 32k rows, backward of the half 541
// against 162; d = 1024, d_e = 512, n = 8, 8k rows 107 against 109, 32k rows 267 against 245.  The lines lie where the two were
// equal over 1176 problems (n 2 to 24, d 512 to 4096, d_e 256 to 2048, 256 to 16384 rows per expert, gathered and copied):
// tiles per SM, and the bytes of the two operands that are d wide.  Widths that are no multiple of 256 have 128-wide whole tiles,
// a fifth slower out of L2.
bool wgrad_whole(const Dims& D) {
    if (wgrad_large(D.n, D.d, D.d_e)) return true;
    const bool copies = !can_fuse_gather(D);
    if (!copies && !wgrad_whole_can_gather(D.l_p)) return false;      // (copying the rows costs more)
    auto tiles = [&](int M, int N) { return (long long)D.n * (M / 128) * (N / (N % 256 == 0 ? 256 : 128)); };
    const double per_sm = (double)(tiles(D.d, D.d_e) + tiles(D.d_e, D.d)) / sm_count();
    const double mb = 2.0 * (copies ? (double)D.Rmax : (double)D.B * D.L) * D.d * D.esize / 1e6;
    if (D.d % 256 == 0 && D.d_e % 256 == 0) return (per_sm >= 1.5 && mb > 64) || (copies && per_sm >= 0.8 && mb > 126);
    return per_sm >= 2.5 && mb > 115;
}

// dy and x gathered inside the consumers' TMA loads (else copied into routed buffers first)
bool bwd_can_gather(const Dims& D) { return can_fuse_gather(D) && (!wgrad_whole(D) || wgrad_whole_can_gather(D.l_p)); }

BwdWs bwd_ws(const Dims& D) {
    WsCarver w;
    w.take(kStatusBytes);
    BwdWs r;
    r.nt = gemm_dg_cols(D.d_e);
    if (r.nt < 1) r.nt = 1;
    r.plan = w.take(plan_bytes(D, true));
    const bool fused = bwd_can_gather(D);      // dy and x gathered inside the consumers' TMA loads
    r.dyg = fused ? 0 : w.take((size_t)D.Rmax * D.d * D.esize);
    r.xg = fused ? 0 : w.take((size_t)D.Rmax * D.d * D.esize);
    r.dh = w.take((size_t)D.Rmax * D.d_e * D.esize);
    r.ag = w.take((size_t)D.Rmax * D.d_e * D.esize);
    r.dxg = w.take((size_t)D.Rmax * D.d * D.esize);
    r.dgp = w.take((size_t)D.Rmax * r.nt * sizeof(float));
    r.G = w.take((size_t)D.B * D.m * D.n * sizeof(float));
    r.rvec = w.take((size_t)D.B * D.m * D.d * sizeof(float));
    r.wpart = w.take((size_t)apply_shape(D).splits * D.d * D.n * sizeof(float));
    const int grads[2][2] = {{D.d_e, D.d}, {D.d, D.d_e}};
    r.wgpart = w.take(wgrad_whole(D) ? 0 : wgrad_stream_scratch_bytes(grads, 2, D.n, D.Rmax));
    r.total = w.off;
    return r;
}

}  // namespace

// Router half of a backward pass, shared by the UoME and SMHA backward: per-row partials of d(loss)/d(gate)
// -> gradient of the router logits G (softmax Jacobians of Eq. 14 and 21) -> partial dW_r (through the pooled token sums)
// and rvec, the vector every real token of a patch receives in dx.  `sum` is the remaining addition over the partials,
// for the caller to hand to launch_combine (which does it beside its own work) or to launch_dwr_sum.
uoe_status launch_router_backward(const Dims& D, const void* x, const void* W_r, const int* expert_idx,
                                  const int* patch_idx, const float* p_samp, const float* p_patch, const PlanPtrs& P,
                                  const float* dgp, int nt, const RouterBwdScratch& rs, float* dW_r, DwrSum* sum,
                                  int* status, cudaStream_t stream, const WReduce& cut) {
    if (!D.bf16) return UOE_ERR_UNSUPPORTED;
    WReduce reduce = cut;
    if (reduce.blocks > 0) reduce.use_threads(router_grad_threads(reduce.by_cut != 0, D.B, (long long)D.k * D.c));
    const size_t smem = ((size_t)2 * D.n * D.m + (size_t)D.k * D.c) * sizeof(float);
    if ((size_t)2 * D.n * D.m * sizeof(float) > 40 * 1024) return UOE_ERR_UNSUPPORTED;
    static SpreadOnce once;
    const uoe_status so = smem_opt_in(once.opt_in, router_grad_kernel, 160 * 1024);      // k c <= n m: at most 60 KB
    if (so != UOE_OK) return so;
    const int grad_ctas = D.B + reduce.blocks;
    {
        ProfScope ps("router_grad", stream);
        launch_k(router_grad_kernel, dim3(grad_ctas), dim3(reduce.threads), spread_smem(once, router_grad_kernel, grad_ctas, smem), stream, dgp, nt, (const int*)P.pair_row, expert_idx, patch_idx,
                 p_samp, p_patch, D.n, D.k, D.m, D.c, D.l_p, D.Lv, rs.G, D.B, reduce);
    }
    UOE_LAUNCHED();
    const ApplyShape a = apply_shape(D);
    const uoe_status st = launch_router_apply<false>(D, a, x, W_r, rs.G, rs.rvec, rs.wpart, nullptr, status, stream);
    if (st != UOE_OK) return st;
    UOE_LAUNCHED();
    *sum = DwrSum{rs.wpart, dW_r, D.d * D.n, a.splits};
    return UOE_OK;
}

uoe_status launch_dwr_sum(const DwrSum& sum, cudaStream_t s) {
    ProfScope ps("dW_r_sum", s);
    launch_k(dwr_sum_kernel, dim3((dwr_sum_items(sum) + kDwrThreads / 32 - 1) / (kDwrThreads / 32)), dim3(kDwrThreads), 0, s, sum);
    UOE_LAUNCHED();
    return UOE_OK;
}

size_t router_backward_scratch_bytes(const Dims& D) {
    return align_up((size_t)D.B * D.m * D.n * 4, 1024) + align_up((size_t)D.B * D.m * D.d * 4, 1024) +
           align_up((size_t)apply_shape(D).splits * D.d * D.n * 4, 1024);
}

RouterBwdScratch router_backward_scratch(const Dims& D, char* base) {
    RouterBwdScratch r;
    r.G = (float*)base;
    base += align_up((size_t)D.B * D.m * D.n * 4, 1024);
    r.rvec = (float*)base;
    base += align_up((size_t)D.B * D.m * D.d * 4, 1024);
    r.wpart = (float*)base;
    return r;
}

size_t mlp_bwd_workspace_bytes(const Dims& D) { return bwd_ws(D).total; }

}  // namespace uoe

using namespace uoe;

extern "C" uoe_status uoe_mlp_backward(const uoe_problem* prob, const void* x, const void* W1, const void* W2,
                                       const void* W_r, const int32_t* expert_idx, const int32_t* patch_idx,
                                       const float* gate, const int32_t* expert_offsets, const float* p_samp,
                                       const float* p_patch, const void* saved_h, const void* dy, void* dx,
                                       float* dW1, float* dW2, float* dW_r, void* ws, size_t ws_bytes,
                                       void* cuda_stream) {
    Dims D;
    uoe_status st = make_dims(prob, D);
    if (st != UOE_OK) return st;
    if (!x || !W1 || !W2 || !W_r || !expert_idx || !patch_idx || !gate || !expert_offsets || !p_samp || !p_patch ||
        !saved_h || !dy || !dx || !dW1 || !dW2 || !dW_r || !ws)
        return UOE_ERR_INVALID_ARG;
    if (D.d_e < 1) return UOE_ERR_INVALID_ARG;
    const void* al[] = {x, W1, W2, saved_h, dy, dx, dW1, dW2, ws};
    for (const void* p : al)
        if (!aligned16(p)) return UOE_ERR_INVALID_ARG;
    // tensor-core path only: bf16, widths that tile the 128-row weight-gradient MMA
    if (!D.bf16 || D.d % 128 != 0 || D.d_e % 128 != 0) return UOE_ERR_UNSUPPORTED;
    if ((size_t)2 * D.n * D.m * sizeof(float) > 40 * 1024) return UOE_ERR_UNSUPPORTED;
    const BwdWs W = bwd_ws(D);
    if (ws_bytes < W.total) return UOE_ERR_WORKSPACE;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const bool use_gate = (prob->flags & UOE_FLAG_GATE) != 0;
    const bool residual = (prob->flags & UOE_FLAG_RESIDUAL) != 0;
    char* base = (char*)ws;
    int* status = (int*)base;
    const PlanPtrs P = plan_ptrs(D, base + W.plan, true);
    void *dyg = base + W.dyg, *xg = base + W.xg, *dh = base + W.dh, *ag = base + W.ag, *dxg = base + W.dxg;
    float* dgp = (float*)(base + W.dgp);
    float* G = (float*)(base + W.G);
    float* rvec = (float*)(base + W.rvec);
    float* wpart = (float*)(base + W.wpart);

    st = launch_plan(D, expert_idx, patch_idx, gate, expert_offsets, P, status, stream, use_gate);
    if (st != UOE_OK) return st;
    // Eq. 18 for dy and x: either inside the TMA loads of the kernels that consume them, or as routed copies
    const bool fused = bwd_can_gather(D);
    if (!fused) {
        st = launch_gather(D, dy, patch_idx, expert_offsets, P, dyg, stream);
        if (st != UOE_OK) return st;
        st = launch_gather(D, x, patch_idx, expert_offsets, P, xg, stream);
        if (st != UOE_OK) return st;
    }
    GemmArgs ga{dyg, W2, nullptr, dh, nullptr, expert_offsets, D.n, D.d, D.d_e, prob->act, true, D.Rmax};
    ga.label = "bwd_da_dh";
    ga.bwd = true; ga.bwd_h = saved_h; ga.row_gate = P.row_gate; ga.row_valid = P.row_valid; ga.dg_part = dgp; ga.C1 = ag;
    if (fused) { ga.gather_x = dy; ga.src_patch = P.src_patch; ga.l_p = D.l_p; ga.Bm = D.B * D.m; }
    st = launch_gemm_bf16(ga, status, stream);
    if (st != UOE_OK) return st;
    // dW2 = ag^T dy_g, dW1 = x_g^T dh
    WReduce reduce;
    if (wgrad_whole(D)) {
        WgradGather gq, gp;
        if (fused) {
            gq.gather_q = true; gq.src_patch = P.src_patch; gq.l_p = D.l_p; gq.Bm = D.B * D.m;
            gp.gather_p = true; gp.src_patch = P.src_patch; gp.l_p = D.l_p; gp.Bm = D.B * D.m;
        }
        st = launch_wgrad_whole(ag, fused ? dy : dyg, dW2, expert_offsets, D.n, D.d_e, D.d, D.Rmax, "wgrad_W2", status, stream, gq);
        if (st != UOE_OK) return st;
        st = launch_wgrad_whole(fused ? x : xg, dh, dW1, expert_offsets, D.n, D.d, D.d_e, D.Rmax, "wgrad_W1", status, stream, gp);
    } else {
        const WStreamProblem probs[2] = {{ag, fused ? dy : dyg, D.d_e, D.d, false, fused, {dW2, nullptr, nullptr}, D.d, false},
                                         {fused ? x : xg, dh, D.d, D.d_e, fused, false, {dW1, nullptr, nullptr}, D.d_e, false}};
        st = launch_wgrad_stream(probs, 2, expert_offsets, D.n, D.Rmax, P.src_patch, D.l_p, D.B * D.m, (float*)(base + W.wgpart),
                                 "wgrad_mlp", status, stream, &reduce);
    }
    if (st != UOE_OK) return st;
    // patches of 128 tokens: dx_g and the combine are one kernel walked by output patch, after the router's term is known
    const bool patch_major = gemm2_patch_can(D, P, nullptr);
    if (!patch_major) {
        GemmArgs gx{dh, W1, nullptr, dxg, nullptr, expert_offsets, D.n, D.d_e, D.d, UOE_ACT_IDENTITY, true, D.Rmax};
        gx.label = "bwd_dx";
        st = launch_gemm_bf16(gx, status, stream);
        if (st != UOE_OK) return st;
    }
    DwrSum sum;
    if (use_gate) {
        RouterBwdScratch rs{G, rvec, wpart};
        st = launch_router_backward(D, x, W_r, expert_idx, patch_idx, p_samp, p_patch, P, dgp, W.nt, rs, dW_r, &sum, status, stream, reduce);
        if (st != UOE_OK) return st;
    } else {
        UOE_CUDA_OK(cudaMemsetAsync(dW_r, 0, (size_t)D.d * D.n * sizeof(float), stream));
        st = launch_wgrad_reduce(reduce, stream);
        if (st != UOE_OK) return st;
    }
    // dx = dy (selective residual) + the routed input gradients (the gate is already inside dh) + router term
    if (patch_major) {
        if (use_gate) st = launch_dwr_sum(sum, stream);
        if (st != UOE_OK) return st;
        return launch_gemm2_patch(D, dh, W1, dy, dx, expert_offsets, P, residual, status, stream, true,
                                  use_gate ? rvec : nullptr, "bwd_dx");
    }
    return launch_combine(D, dy, dxg, P, residual, false, dx, stream, use_gate ? rvec : nullptr, sum);
}


namespace uoe {
size_t balance_bwd_workspace_bytes(const Dims& D) { return kStatusBytes + router_backward_scratch_bytes(D); }
}  // namespace uoe

extern "C" uoe_status uoe_route_balance_backward(const uoe_problem* prob, const void* x, const void* W_r,
                                                 const float* p_patch, float alpha, const float* dloss, void* dx,
                                                 float* dW_r, void* ws, size_t ws_bytes, void* cuda_stream) {
    Dims D;
    uoe_status st = make_dims(prob, D);
    if (st != UOE_OK) return st;
    if (!x || !W_r || !p_patch || !dloss || !dx || !dW_r || !ws) return UOE_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(dx) || !aligned16(ws)) return UOE_ERR_INVALID_ARG;
    if (!D.bf16) return UOE_ERR_UNSUPPORTED;
    if ((size_t)D.n * D.m * sizeof(float) > 36 * 1024) return UOE_ERR_UNSUPPORTED;
    if (ws_bytes < balance_bwd_workspace_bytes(D)) return UOE_ERR_WORKSPACE;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const RouterBwdScratch rs = router_backward_scratch(D, (char*)ws + kStatusBytes);
    {
        ProfScope ps("balance_bwd", stream);
        launch_k(balance_bwd_kernel, dim3(D.B), dim3(kBalanceThreads), (size_t)D.n * (D.m + 1) * sizeof(float), stream, p_patch, dloss, D.Lv, D.n,
                 D.k, D.m, D.l_p, alpha, rs.G);
    }
    UOE_LAUNCHED();
    const ApplyShape a = apply_shape(D);
    st = launch_router_apply<true>(D, a, x, W_r, rs.G, nullptr, rs.wpart, dx, (int*)ws, stream);
    if (st != UOE_OK) return st;
    UOE_LAUNCHED();
    return launch_dwr_sum(DwrSum{rs.wpart, dW_r, D.d * D.n, a.splits}, stream);
}
