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

namespace uoe {
namespace {

constexpr int kThreads = 256;

// Gradient of the router logits of one sample from the per-row gate gradients.  grid B, 512 threads, dynamic shared
// memory (2 n m + k c) floats.  A warp per slab adds the slab's per-row, per-column-tile partials (fixed order), then the
// softmax Jacobians of Eq. 14 and 21:  G[b,j,i] = dlogit_patch[b,i,j]/cnt_j + dlogit_samp[b,i]/L_valid.
// Latency-bound (a sample's partials are a few KB to a few hundred KB); one launch instead of a slab-sum kernel and a
// Jacobian kernel whose sums over a slot list were one thread's serial loop.
constexpr int kGradThreads = kReduceThreads;
__global__ void __launch_bounds__(kGradThreads, 2)
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
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int idx = tid; idx < n * m; idx += kGradThreads) { pp[idx] = p_patch[(size_t)b * n * m + idx]; dpp[idx] = 0.f; }
    if (tid < 32) { ps[tid] = tid < n ? p_samp[(size_t)b * n + tid] : 0.f; dps[tid] = 0.f; }
    const int len = l_p * nt;
    for (int slab = warp; slab < k * c; slab += kGradThreads / 32) {
        const int j = patch_idx[(size_t)b * k * c + slab];
        float a = 0.f;
        if (j >= 0 && j < m) {
            const float* src = dg_part + ((size_t)pair_row[b * k + slab / c] + (size_t)(slab % c) * l_p) * nt;
            int q = lane;
            for (; q + 96 < len; q += 128) {
                const float t0 = src[q], t1 = src[q + 32], t2 = src[q + 64], t3 = src[q + 96];
                a += (t0 + t1) + (t2 + t3);
            }
            for (; q < len; q += 32) a += src[q];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) dg[slab] = a;
    }
    __syncthreads();
    // gate = P_samp * P_patch: a warp per chosen expert, lanes over its slots
    for (int s = warp; s < k; s += kGradThreads / 32) {
        const int i = expert_idx[(size_t)b * k + s];
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
    for (int j = tid; j < m; j += kGradThreads) {         // softmax Jacobian of each patch gate (Eq. 14)
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
// Bound by reading x once.  Grid (column blocks, splits), two CTAs per SM in all; a CTA has one thread per column of its
// block and walks batches of eight slices: slice = (unit, row thread), where a unit is a patch or a segment of at most
// 64 rows of a longer one, 16-byte loads, about eight rows per thread and batch, so a batch is 8 / RT units whose rows
// are dealt to RT row threads.  The next batch's loads are in flight under this batch's arithmetic.  The sums meet in shared memory, then a thread adds its column's products: the pooled tensor
// never reaches memory.  Every split leaves its own partial dW_r (dwr_sum adds them in split order).  SPREAD: the vector
// is written to every row of dx at once instead of to rvec (the balance loss, whose whole dx it is).
// Against a pooling kernel, one or two product kernels, a vector kernel and a spreading kernel (us, cold caches):
// 23 instead of 58 at B = 256, L = 224, d = 384, n = 6;  9 instead of 22 at B = 16, L = 512, d = 512, n = 8;  77 as before
// at B = 8, L = 4096, d = 4096, n = 16 (3.9 TB/s: two CTAs per SM do not cover the batch hand-offs there);  SPREAD 39
// instead of 84 at B = 16, L = 2048, d = 1024, n = 16.
constexpr int kSlices = 8;
template <int NMAX, bool SPREAD>
__global__ void __launch_bounds__(320, NMAX > 16 ? 1 : 2)
router_apply_kernel(const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ W_r, const float* __restrict__ G,
                    float* __restrict__ rvec, float* __restrict__ part, __nv_bfloat16* __restrict__ dx, int units, int L, int Lv,
                    int d, int n, int m, int l_p, int nseg, int RT, int batches_per_cta) {
    pdl_trigger();
    extern __shared__ float s_pool[];                // [kSlices][CW] column sums; SPREAD: then [kSlices / RT][CW] bfloat16
    __shared__ float sG[kSlices * NMAX];
    const int CW = blockDim.x, tid = threadIdx.x;    // CW: a multiple of 64
    const int c0 = blockIdx.x * CW;
    const int ct = tid % (CW / 8), slice = tid / (CW / 8);
    const int PB = kSlices / RT;                     // units per batch
    const int seg_rows = (l_p + nseg - 1) / nseg;
    const int my_q = slice / RT, my_rt = slice % RT;
    const int col = c0 + ct * 8, dd = c0 + tid;
    pdl_wait();
    float acc[NMAX], w[NMAX];
#pragma unroll
    for (int i = 0; i < NMAX; ++i) {
        acc[i] = 0.f;
        w[i] = (i < n && dd < d) ? __bfloat162float(W_r[(size_t)dd * n + i]) : 0.f;
    }
    const int q_lo = blockIdx.y * batches_per_cta * PB, q_hi = min(units, q_lo + batches_per_cta * PB);
    // the loads of a batch: this thread's first eight rows, and its share of the batch's G (at most four values)
    uint4 ld[8];
    float gv[4];
    int rows = 0, rows_all = 0;                     // real rows of the unit, all its rows
    const __nv_bfloat16* base = nullptr;
    auto issue = [&](int q0) {
        rows = rows_all = 0;
        const int unit = q0 + my_q;
        if (my_q < PB && unit < q_hi && col < d) {
            const int bj = nseg == 1 ? unit : unit / nseg, b = bj / m, s0 = nseg == 1 ? 0 : (unit - bj * nseg) * seg_rows;
            const int r0 = (bj - b * m) * l_p + s0;      // first row in the sample
            rows_all = min(seg_rows, l_p - s0);
            rows = max(0, min(rows_all, Lv - r0));
            base = x + ((size_t)b * L + r0) * d + col;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (my_rt + u * RT < rows) ld[u] = ld_stream16(base + (size_t)(my_rt + u * RT) * d);
        const int ng = min(PB, q_hi - q0) * n;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (tid + u * CW < ng)
                gv[u] = nseg == 1 ? G[(size_t)q0 * n + tid + u * CW] : G[(size_t)((q0 + (tid + u * CW) / n) / nseg) * n + (tid + u * CW) % n];
    };
    if (q_lo < q_hi) issue(q_lo);
    for (int q0 = q_lo; q0 < q_hi; q0 += PB) {
        const int nb = min(PB, q_hi - q0), rows_q = rows, rows_all_q = rows_all;
        __nv_bfloat16* dx_base = SPREAD ? dx + (base - x) : nullptr;
        {   // ---- column sums of this thread's slice ----
            float cs[8];
#pragma unroll
            for (int v = 0; v < 8; ++v) cs[v] = 0.f;
            auto add = [&](const uint4& t) {
                float f[8];
                unpack16<__nv_bfloat16>(t, f);
#pragma unroll
                for (int v = 0; v < 8; ++v) cs[v] += f[v];
            };
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (my_rt + u * RT < rows) add(ld[u]);
            int r = my_rt + 8 * RT;
            for (; r + 3 * RT < rows; r += 4 * RT) {
                uint4 t[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) t[u] = ld_stream16(base + (size_t)(r + u * RT) * d);
#pragma unroll
                for (int u = 0; u < 4; ++u) add(t[u]);
            }
            for (; r < rows; r += RT) add(ld_stream16(base + (size_t)r * d));
#pragma unroll
            for (int v = 0; v < 8; v += 4)
                *(float4*)(s_pool + slice * CW + ct * 8 + v) = make_float4(cs[v], cs[v + 1], cs[v + 2], cs[v + 3]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int idx = tid + u * CW;
            if (idx < nb * n) sG[(idx / n) * NMAX + idx % n] = gv[u];
        }
        __syncthreads();
        if (q0 + PB < q_hi) issue(q0 + PB);
        float rv[kSlices];
#pragma unroll
        for (int q = 0; q < kSlices; ++q) {          // (unrolled over the largest batch so that rv stays in registers)
            rv[q] = 0.f;
            if (q < nb) {
                float p = 0.f;
                for (int rt = 0; rt < RT; ++rt) p += s_pool[(q * RT + rt) * CW + tid];
                float a = 0.f;
#pragma unroll
                for (int i = 0; i < NMAX; ++i) {
                    if (i < n) {
                        const float g = sG[q * NMAX + i];
                        acc[i] = fmaf(p, g, acc[i]);
                        a = fmaf(w[i], g, a);
                    }
                }
                rv[q] = a;
                if (!SPREAD && dd < d && (nseg == 1 || (q0 + q) % nseg == 0)) rvec[(size_t)(nseg == 1 ? q0 + q : (q0 + q) / nseg) * d + dd] = a;
            }
        }
        __syncthreads();
        if (SPREAD) {
            __nv_bfloat16* s_rv = (__nv_bfloat16*)s_pool;
#pragma unroll
            for (int q = 0; q < kSlices; ++q)
                if (q < nb) s_rv[q * CW + tid] = __float2bfloat16(rv[q]);
            __syncthreads();
            if (my_q < nb && col < d) {
                const uint4 v = *(const uint4*)(s_rv + my_q * CW + ct * 8);
                for (int r = my_rt; r < rows_all_q; r += RT) st_stream16(dx_base + (size_t)r * d, r < rows_q ? v : make_uint4(0, 0, 0, 0));
            }
            __syncthreads();
        }
    }
    if (dd < d) {
#pragma unroll
        for (int i = 0; i < NMAX; ++i)
            if (i < n) part[((size_t)blockIdx.y * d + dd) * n + i] = acc[i];
    }
}

__global__ void __launch_bounds__(kThreads)
dwr_sum_kernel(const DwrSum s) {
    pdl_trigger();
    pdl_wait();
    dwr_sum(s, blockIdx.x);
}

// Column block, row threads and splits of router_apply_kernel for a problem.
struct ApplyShape { int CW, RT, nseg, col_blocks, splits, per; };
ApplyShape apply_shape(const Dims& D) {
    ApplyShape a;
    a.CW = D.d < 256 ? (D.d + 63) / 64 * 64 : 256;
    for (int cw : {256, 320, 192, 128})
        if (D.d % cw == 0) { a.CW = cw; break; }
    a.col_blocks = (D.d + a.CW - 1) / a.CW;
    // rows of a patch are dealt to as many threads as leave each about eight rows, one batch of loads
    a.nseg = (D.l_p + 63) / 64;
    a.RT = 1;
    while (a.RT < kSlices && (D.l_p + a.nseg - 1) / a.nseg >= 16 * a.RT) a.RT *= 2;
    const int PB = kSlices / a.RT, batches = (D.B * D.m * a.nseg + PB - 1) / PB;
    const int cap = 2 * 148 / a.col_blocks > 1 ? 2 * 148 / a.col_blocks : 1;        // two CTAs per SM: one full wave
    a.splits = batches < cap ? batches : cap;
    a.per = (batches + a.splits - 1) / a.splits;
    a.splits = (batches + a.per - 1) / a.per;
    return a;
}
template <bool SPREAD>
void launch_router_apply(const Dims& D, const ApplyShape& a, const void* x, const void* W_r, const float* G, float* rvec,
                         float* part, void* dx, cudaStream_t s) {
    auto go = [&](SpreadOnce& once, auto kern) {
        const size_t smem = spread_smem(once, kern, (long long)a.col_blocks * a.splits, (size_t)kSlices * a.CW * sizeof(float));
        launch_k(kern, dim3(a.col_blocks, a.splits), dim3(a.CW), smem, s, (const __nv_bfloat16*)x,
                 (const __nv_bfloat16*)W_r, G, rvec, part, (__nv_bfloat16*)dx, D.B * D.m * a.nseg, D.L, D.Lv, D.d, D.n, D.m, D.l_p, a.nseg,
                 a.RT, a.per);
    };
    ProfScope ps("router_apply", s);
    static SpreadOnce once[3];
    if (D.n <= 8) go(once[0], router_apply_kernel<8, SPREAD>);
    else if (D.n <= 16) go(once[1], router_apply_kernel<16, SPREAD>);
    else go(once[2], router_apply_kernel<32, SPREAD>);
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

// dy and x gathered inside the consumers' TMA loads (else copied into routed buffers first)
bool bwd_can_gather(const Dims& D) {
    return can_fuse_gather(D) && (!wgrad_large(D.n, D.d, D.d_e) || wgrad_large_can_gather(D.l_p));
}

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
    r.wgpart = w.take(wgrad_large(D.n, D.d, D.d_e) ? 0 : wgrad_stream_scratch_bytes());
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
                                  cudaStream_t stream, const WReduce& reduce) {
    if (!D.bf16) return UOE_ERR_UNSUPPORTED;
    const size_t smem = ((size_t)2 * D.n * D.m + (size_t)D.k * D.c) * sizeof(float);
    if ((size_t)2 * D.n * D.m * sizeof(float) > 40 * 1024) return UOE_ERR_UNSUPPORTED;
    static SpreadOnce once;
    const uoe_status so = smem_opt_in(once.opt_in, router_grad_kernel, 160 * 1024);      // k c <= n m: at most 60 KB
    if (so != UOE_OK) return so;
    const int grad_ctas = D.B + reduce.blocks;
    {
        ProfScope ps("router_grad", stream);
        launch_k(router_grad_kernel, dim3(grad_ctas), dim3(kGradThreads), spread_smem(once, router_grad_kernel, grad_ctas, smem), stream, dgp, nt, (const int*)P.pair_row, expert_idx, patch_idx,
                 p_samp, p_patch, D.n, D.k, D.m, D.c, D.l_p, D.Lv, rs.G, D.B, reduce);
    }
    UOE_LAUNCHED();
    const ApplyShape a = apply_shape(D);
    launch_router_apply<false>(D, a, x, W_r, rs.G, rs.rvec, rs.wpart, nullptr, stream);
    UOE_LAUNCHED();
    *sum = DwrSum{rs.wpart, dW_r, D.d * D.n, a.splits};
    return UOE_OK;
}

uoe_status launch_dwr_sum(const DwrSum& sum, cudaStream_t s) {
    ProfScope ps("dW_r_sum", s);
    launch_k(dwr_sum_kernel, dim3(dwr_sum_blocks(sum)), dim3(kThreads), 0, s, sum);
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
    if (wgrad_large(D.n, D.d, D.d_e)) {
        WgradGather gq, gp;
        if (fused) {
            gq.gather_q = true; gq.src_patch = P.src_patch; gq.l_p = D.l_p; gq.Bm = D.B * D.m;
            gp.gather_p = true; gp.src_patch = P.src_patch; gp.l_p = D.l_p; gp.Bm = D.B * D.m;
        }
        st = launch_wgrad_large(ag, fused ? dy : dyg, dW2, expert_offsets, D.n, D.d_e, D.d, D.Rmax, "wgrad_W2", status, stream, gq);
        if (st != UOE_OK) return st;
        st = launch_wgrad_large(fused ? x : xg, dh, dW1, expert_offsets, D.n, D.d, D.d_e, D.Rmax, "wgrad_W1", status, stream, gp);
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
        st = launch_router_backward(D, x, W_r, expert_idx, patch_idx, p_samp, p_patch, P, dgp, W.nt, rs, dW_r, &sum, stream, reduce);
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
    launch_router_apply<true>(D, a, x, W_r, rs.G, nullptr, rs.wpart, dx, stream);
    UOE_LAUNCHED();
    return launch_dwr_sum(DwrSum{rs.wpart, dW_r, D.d * D.n, a.splits}, stream);
}
