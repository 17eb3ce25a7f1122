// uoe_smha_backward: gradients of sum(y * dy) for y = uoe_smha_forward(x, ...) with the selection held constant
// (derivative of Eq. 27-36; with gating also of Eq. 14 and 21 through the gate weights).  The paper gives no
// backward text.  Nothing is saved by the forward: q, k, v, o and the log-sum-exp are recomputed here.
//
// In routed-row space, for the rows r of pair (b, i) with combine weight w_r (0 on pad-token rows):
//   q, k, v = x_g W^{q,k,v}_i ; o, lse = attention(q, k, v)              recomputed (Eq. 28-34)
//   do_raw  = dy_g W^o_i^T                                               grouped GEMM (K-major weights), whose epilogue makes
//   dgate(patch) = sum_r <do_raw_r, o_r> ;  do = w do_raw ; og = w o ;  delta_{r,h} = sum_{c in head h} do o (do as rounded)
//             (as a kernel of its own this was another pass over do_raw, o, do and og: 20 us for the image block, B = 256)
//   dq, dk, dv = attention backward(q, k, v, do, lse, delta)             -> one buffer [rows, 3 d_g]
//   dx_g = [dq dk dv] [W^q_i W^k_i W^v_i]^T                              one grouped GEMM, K = 3 d_g, weights read in place
//   d[W^q W^k W^v]_i = x_g^T [dq dk dv] ;  dW^o_i^T = dy_g^T og          ragged-K weight-gradient GEMMs
// then dx = dy + combine(dx_g) + router term, and the router gradients as in the UoME backward.
#include "kernels.cuh"

namespace uoe {

uoe_status launch_attention(const Dims& D, const void* q, const void* k, const void* v, void* o, float* lse,
                            const int* pair_row, const int* patch_idx, bool causal, int* status, cudaStream_t s,
                            const void* Wo = nullptr, const int* expert_idx = nullptr, void* z = nullptr);
bool attention_can_fuse_out(const Dims& D);
uoe_status launch_attention_backward(const Dims& D, const void* q, const void* k, const void* v, const void* dout,
                                     const float* lse, const float* delta, void* dq, void* dk, void* dv, int ld_out,
                                     const int* pair_row, const int* patch_idx, bool causal, const Rope& rope, int* status,
                                     cudaStream_t s);

namespace {

struct SmhaBwdWs {
    size_t plan, xg, dyg, q, k, v, o, dout, og, dqkv, dxg, lse, delta, dgp, router, wgpart, total;
};

SmhaBwdWs smha_bwd_ws(const Dims& D) {
    WsCarver w;
    w.take(kStatusBytes);
    SmhaBwdWs r;
    const int heads = D.d_g > 0 ? D.d_g / 64 : 1;
    const size_t rg = (size_t)D.Rmax * D.d_g * D.esize;
    r.plan = w.take(plan_bytes(D, true));
    const bool fused = can_fuse_gather(D);      // x and dy gathered inside the consumers' TMA loads
    r.xg = fused ? 0 : w.take((size_t)D.Rmax * D.d * D.esize);
    r.dyg = fused ? 0 : w.take((size_t)D.Rmax * D.d * D.esize);
    r.q = w.take(rg); r.k = w.take(rg); r.v = w.take(rg); r.o = w.take(rg); r.dout = w.take(rg); r.og = w.take(rg);
    r.dqkv = w.take(3 * rg);
    r.dxg = w.take((size_t)D.Rmax * D.d * D.esize);
    r.lse = w.take((size_t)D.Rmax * heads * 4);
    r.delta = w.take((size_t)D.Rmax * heads * 4);
    r.dgp = w.take((size_t)D.Rmax * heads * 4);
    r.router = w.take(router_backward_scratch_bytes(D));
    const int grads[2][2] = {{D.d, 3 * D.d_g}, {D.d, D.d_g}};
    r.wgpart = w.take(wgrad_stream_scratch_bytes(grads, 2, D.n, D.Rmax));
    r.total = w.off;
    return r;
}

}  // namespace

size_t smha_bwd_workspace_bytes(const Dims& D) { return smha_bwd_ws(D).total; }

}  // namespace uoe

using namespace uoe;

extern "C" uoe_status uoe_smha_backward(const uoe_problem* prob, const void* x, const void* Wq, const void* Wk,
                                        const void* Wv, const void* Wo, const void* W_r, const int32_t* expert_idx,
                                        const int32_t* patch_idx, const float* gate, const int32_t* expert_offsets,
                                        const float* p_samp, const float* p_patch, const void* dy, void* dx,
                                        float* dWq, float* dWk, float* dWv, float* dWo, float* dW_r, void* ws,
                                        size_t ws_bytes, void* cuda_stream) {
    Dims D;
    uoe_status st = make_dims(prob, D);
    if (st != UOE_OK) return st;
    if (!x || !Wq || !Wk || !Wv || !Wo || !W_r || !expert_idx || !patch_idx || !gate || !expert_offsets || !p_samp ||
        !p_patch || !dy || !dx || !dWq || !dWk || !dWv || !dWo || !dW_r || !ws)
        return UOE_ERR_INVALID_ARG;
    if (D.H < 1 || D.d_g < 1) return UOE_ERR_INVALID_ARG;
    const void* al[] = {x, Wq, Wk, Wv, Wo, dy, dx, dWq, dWk, dWv, dWo, ws};
    for (const void* p : al)
        if (!aligned16(p)) return UOE_ERR_INVALID_ARG;
    // tensor-core path only: bf16, 64-wide heads, model width that tiles the 128-row weight-gradient MMA
    if (!D.bf16 || D.d_h != 64 || D.d % 128 != 0) return UOE_ERR_UNSUPPORTED;
    if ((long long)D.B * D.k > 65535) return UOE_ERR_UNSUPPORTED;  // grids carry the pairs on an axis of this extent (y in the attention backward)
    const SmhaBwdWs W = smha_bwd_ws(D);
    if (ws_bytes < W.total) return UOE_ERR_WORKSPACE;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const bool use_gate = (prob->flags & UOE_FLAG_GATE) != 0;
    const bool residual = (prob->flags & UOE_FLAG_RESIDUAL) != 0;
    const bool causal = (prob->flags & UOE_FLAG_CAUSAL) != 0;
    const int heads = D.d_g / 64;
    char* base = (char*)ws;
    int* status = (int*)base;
    const PlanPtrs P = plan_ptrs(D, base + W.plan, true);
    void *xg = base + W.xg, *dyg = base + W.dyg, *q = base + W.q, *k = base + W.k, *v = base + W.v, *o = base + W.o;
    void *dout = base + W.dout, *og = base + W.og, *dqkv = base + W.dqkv, *dxg = base + W.dxg;
    float *lse = (float*)(base + W.lse), *delta = (float*)(base + W.delta), *dgp = (float*)(base + W.dgp);
    const RouterBwdScratch rs = router_backward_scratch(D, base + W.router);
    const long long rowb = (long long)D.d_g * D.esize;

    st = launch_plan(D, expert_idx, patch_idx, gate, expert_offsets, P, status, stream, use_gate, PlanTails{{q, k, v, dout}, rowb});
    if (st != UOE_OK) return st;
    // Eq. 18 for x and dy: either inside the TMA loads of the kernels that consume them, or as routed copies
    const bool fused = can_fuse_gather(D);
    if (!fused) {
        st = launch_gather(D, x, patch_idx, expert_offsets, P, xg, stream);
        if (st != UOE_OK) return st;
        st = launch_gather(D, dy, patch_idx, expert_offsets, P, dyg, stream);
        if (st != UOE_OK) return st;
    }

    // ---- forward recomputation (Eq. 28-34) ----
    const Rope rope = rope_of(D, P, patch_idx);      // Eq. 32 (nothing if d_rope = 0)
    if (smha_can_fuse(D, true)) {
        SmhaFused f;
        f.x = x; f.W[0] = Wq; f.W[1] = Wk; f.W[2] = Wv; f.q = q; f.k = k; f.v = v; f.o = o; f.lse = lse;
        st = launch_smha_fused(D, f, P, patch_idx, expert_idx, expert_offsets, causal, rope, status, stream);
        if (st != UOE_OK) return st;
    } else {
        GemmArgs gq{xg, Wq, nullptr, q, nullptr, expert_offsets, D.n, D.d, D.d_g, UOE_ACT_IDENTITY, false, D.Rmax};
        if (fused) { gq.gather_x = x; gq.src_patch = P.src_patch; gq.l_p = D.l_p; gq.Bm = D.B * D.m; }
        gq.label = "qkv_proj";
        gq.nmat = 3; gq.W1 = Wk; gq.W2 = Wv; gq.C1 = k; gq.C2 = v;
        gq.rope = &rope;
        st = launch_gemm_bf16(gq, status, stream);
        if (st != UOE_OK) return st;
        st = launch_attention(D, q, k, v, o, lse, P.pair_row, patch_idx, causal, status, stream);
        if (st != UOE_OK) return st;
    }

    // ---- out-projection backward ----
    GemmArgs gd{dyg, Wo, nullptr, dout, nullptr, expert_offsets, D.n, D.d, D.d_g, UOE_ACT_IDENTITY, true, D.Rmax};
    if (fused) { gd.gather_x = dy; gd.src_patch = P.src_patch; gd.l_p = D.l_p; gd.Bm = D.B * D.m; }
    gd.label = "bwd_do";
    // with the raw gradient still in float32: its product with o, the gated do and o, zeroed padding rows of dq, dk, dv
    gd.bwd_h = o; gd.row_gate = P.row_gate; gd.row_valid = P.row_valid; gd.dg_part = dgp; gd.C1 = og;
    gd.att = AttBwd{delta, P.expert_end, (__nv_bfloat16*)dqkv};
    st = launch_gemm_bf16(gd, status, stream);
    if (st != UOE_OK) return st;

    // ---- attention backward ----
    __nv_bfloat16* dq = (__nv_bfloat16*)dqkv;
    st = launch_attention_backward(D, q, k, v, dout, lse, delta, dq, dq + D.d_g, dq + 2 * D.d_g, 3 * D.d_g, P.pair_row,
                                   patch_idx, causal, rope, status, stream);
    if (st != UOE_OK) return st;

    // ---- projection backward: dx_g and the q/k/v weight gradients from the concatenated [dq dk dv] ----
    GemmArgs gx{dqkv, Wq, nullptr, dxg, nullptr, expert_offsets, D.n, 3 * D.d_g, D.d, UOE_ACT_IDENTITY, true, D.Rmax};
    gx.k_mats = 3; gx.W1 = Wk; gx.W2 = Wv;      // K block by K block from the three weight tensors
    gx.label = "bwd_dx_att";
    st = launch_gemm_bf16(gx, status, stream);
    if (st != UOE_OK) return st;
    // d[W^q W^k W^v] = x_g^T [dq dk dv], column blocks straight to the three outputs; dW^o^T = dy_g^T og, written transposed
    WReduce reduce;
    const WStreamProblem probs[2] = {{fused ? x : xg, dqkv, D.d, 3 * D.d_g, fused, false, {dWq, dWk, dWv}, D.d_g, false},
                                     {fused ? dy : dyg, og, D.d, D.d_g, fused, false, {dWo, nullptr, nullptr}, D.d_g, true}};
    st = launch_wgrad_stream(probs, 2, expert_offsets, D.n, D.Rmax, P.src_patch, D.l_p, D.B * D.m, (float*)(base + W.wgpart),
                             "wgrad_att", status, stream, &reduce);
    if (st != UOE_OK) return st;

    // ---- router ----
    DwrSum sum;
    if (use_gate) {
        st = launch_router_backward(D, x, W_r, expert_idx, patch_idx, p_samp, p_patch, P, dgp, heads, rs, dW_r, &sum, status, stream, reduce);
        if (st != UOE_OK) return st;
    } else {
        UOE_CUDA_OK(cudaMemsetAsync(dW_r, 0, (size_t)D.d * D.n * sizeof(float), stream));
        st = launch_wgrad_reduce(reduce, stream);
        if (st != UOE_OK) return st;
    }
    return launch_combine(D, dy, dxg, P, residual, false, dx, stream, use_gate ? rs.rvec : nullptr, sum);
}
