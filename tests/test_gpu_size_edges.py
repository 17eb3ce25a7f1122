"""GPU parity at the sizes where a kernel's tiling, split or dispatch can go wrong: tile edges, remainders, the smallest
and largest of a range.  References: the float64 oracle on the GPU's own selection.

Tolerances: bfloat16 results max|err| <= 2e-2 * max|ref| (operands carry 2^-9 relative rounding through three to four
roundings, a few 1e-3 of the output scale; see the other parity tests).
"""
import numpy as np
import pytest
import torch

import uoe_inputs as gen
from oracle import uoe_oracle as orc
from tests.helpers import problem_of, rel_inf, to_dev, to_f64

pytestmark = pytest.mark.gpu

TOL = 2e-2


def _att(**kw):
    base = dict(B=3, L=96, L_valid=96, m=6, c=3, d=64, n=2, k=1, d_ff=0, H=2, d_h=64, dtype="bf16", w_std=0.08, causal=False)
    base.update(kw)
    return gen.tiny(**base)


# rotary positions come from the routed row inside the projection: patches that do not divide a tile, several heads,
# whole samples per expert (identity plan), unused slots, and the plan both ways (router-written, plan kernel)
ROPE_CASES = {
    "patch20_two_heads": (_att(B=5, L=140, L_valid=133, m=7, c=4, n=3, k=2, H=6, causal=True), 32, {}),
    "whole_samples": (_att(B=4, L=160, L_valid=150, m=10, c=10, n=4, k=2, H=4), 64, {}),
    "unused_slots": (_att(B=4, L=128, L_valid=128, m=16, c=12, n=4, k=2, H=4), 16, {"dynamic_c": True}),
    "two_heads_many_rows": (_att(B=8, L=1024, L_valid=1010, m=16, c=8, d=192, n=4, k=2, H=8, causal=True), 32, {}),
    "two_heads_many_rows_no_rope": (_att(B=8, L=1024, L_valid=1024, m=16, c=8, d=192, n=4, k=2, H=8), 0, {}),
    "patch1": (_att(B=2, L=40, L_valid=39, m=40, c=17, n=2, k=2, H=2), 2, {}),
}


@pytest.mark.parametrize("entry", ["block", "halves"])
@pytest.mark.parametrize("name", list(ROPE_CASES))
def test_rotary_positions_of_routed_rows(name, entry):
    import paper_2503_02495_b200 as uoe
    w, d_rope, kw = ROPE_CASES[name]
    x, Wr = gen.make_x(w), gen.store(gen.make_router(w, "att").f64 * 20, w.dtype)
    ws = gen.make_attn_weights(w)
    prob = problem_of(w, "att", residual=False, d_rope=d_rope, **kw)
    xd, Wrd, wd = to_dev(x), to_dev(Wr), [to_dev(q) for q in ws]
    if entry == "block":
        r = uoe.alloc_routing(prob)
        y = uoe.uoe_block_forward(prob, None, xd, dict(zip(("Wr_att", "Wq", "Wk", "Wv", "Wo"), [Wrd] + wd)), r_att=r)
    else:
        r = uoe.uoe_route(prob, xd, Wrd)
        y = uoe.uoe_smha_forward(prob, xd, *wd, r)
    ro = orc.with_selection(x.f64, Wr.f64, r.expert_idx.cpu().numpy(), r.patch_idx.cpu().numpy(), w.m, w.L_valid)
    ref = orc.smha_forward(x.f64, *[q.f64 for q in ws], ro, w.d_h, w.causal, residual=False, d_rope=d_rope)
    assert rel_inf(to_f64(y), ref) <= TOL


# one pass over x for dW_r and dx: every column-block width, row segments (patches above 32 rows), one-row patches,
# more experts than the widest register tile but one, a width that no block divides
@pytest.mark.parametrize("kw", [dict(B=2, m=3, L=390, L_valid=301, d=200, n=20, k=5, c=2), dict(B=5, m=33, L=33, L_valid=31, d=640, n=9, k=3, c=8),
                                dict(B=1, m=4, L=64, L_valid=64, d=72, n=3, k=1, c=1), dict(B=40, m=9, L=216, L_valid=216, d=384, n=8, k=2, c=3),
                                dict(B=3, m=2, L=130, L_valid=130, d=2048, n=16, k=4, c=2)],
                         ids=lambda k: f"d{k['d']}n{k['n']}")
def test_router_gradients_of_the_balance_loss(kw):
    """Tolerance: the stored dx is bfloat16 (2^-9), dW_r float32; 2e-2 of the largest value as for the other gradients."""
    import paper_2503_02495_b200 as uoe
    w = gen.tiny(dtype="bf16", d_ff=0, H=0, **kw)
    x, Wr = gen.make_x(w), gen.store(gen.make_router(w).f64 * 20, w.dtype)
    prob = problem_of(w, "mlp")
    xd, Wrd = to_dev(x), to_dev(Wr)
    r = uoe.uoe_route(prob, xd, Wrd)
    dloss = gen.normal(7, 0, (w.B,)).astype(np.float32)
    dx, dWr = uoe.uoe_route_balance_backward(prob, xd, Wrd, r.p_patch, 0.05, torch.from_numpy(dloss).cuda())
    ref_dx, ref_dWr = orc.balance_loss_backward(x.f64, Wr.f64, w.m, w.L_valid, w.k, 0.05, dloss.astype(np.float64))
    assert rel_inf(to_f64(dx), ref_dx) <= TOL
    assert rel_inf(to_f64(dWr), ref_dWr) <= TOL
    assert np.all(to_f64(dx)[:, w.L_valid:] == 0)


# a warp per expert (a second turn past sixteen), 32 patches per step: one expert, one patch, a step of one patch, all experts
@pytest.mark.parametrize("n,k,m,L_valid", [(1, 1, 1, 3), (17, 4, 33, 130), (32, 32, 65, 260), (20, 1, 64, 256), (5, 2, 31, 121)])
def test_loads_and_balance_loss(n, k, m, L_valid):
    """Whole numbers exact on the gate values the GPU wrote; the loss is a float32 sum of at most 65 positive terms in
    shuffle order (65 * 2^-24 = 4e-6 relative)."""
    import paper_2503_02495_b200 as uoe
    w = gen.tiny(B=3, L=4 * m, L_valid=L_valid, m=m, c=1, d=64, n=n, k=k, d_ff=0, H=0, dtype="bf16")
    x, Wr = gen.make_x(w), gen.store(gen.make_router(w).f64 * 20, w.dtype)
    prob = problem_of(w, "mlp")
    r = uoe.uoe_route(prob, to_dev(x), to_dev(Wr))
    lb, cnt, cd = uoe.uoe_route_balance(prob, r.p_patch, alpha=0.01)
    pp = r.p_patch.cpu().numpy().astype(np.float64)
    pc = orc.patch_valid_counts(w.L, w.m, w.L_valid)
    assert np.array_equal(cnt.cpu().numpy(), np.stack([orc.patch_expert_counts(pp[b], pc, k) for b in range(w.B)]))
    assert np.array_equal(cd.cpu().numpy(), orc.dynamic_capacity(pp, pc, k))
    ref = orc.balance_loss(pp, pc, k, alpha=0.01)
    assert np.abs(lb.cpu().numpy() - ref).max() <= 1e-5 * np.abs(ref).max()


def test_more_samples_than_a_grid_dimension_holds():
    """Scores of 65541 samples take two launches, the ticket runs through both.  Tolerance 2e-6: softmax values at most 1 from
    float32 sums of 33 * 16 bfloat16 products (528 * 2^-24 * |logit| below 1, divided by 33 tokens)."""
    import paper_2503_02495_b200 as uoe
    B, L, d, n, k = 65541, 33, 16, 4, 2
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(B, L, d, device="cuda", generator=g).bfloat16()
    Wr = (0.5 * torch.randn(d, n, device="cuda", generator=g)).bfloat16()
    r = uoe.uoe_route(uoe.Problem(B=B, L=L, L_valid=L, d=d, n=n, k=k, m=1, c=1, dtype="bf16"), x, Wr)
    ref = torch.softmax(x.double().mean(1) @ Wr.double(), dim=1)
    assert (r.p_samp.double() - ref).abs().max() <= 2e-6
    assert (r.p_patch.reshape(B, n).double() - ref).abs().max() <= 2e-6
    picked = ref.gather(1, r.expert_idx.long())
    assert (picked.min(1).values >= ref.topk(k, dim=1).values.min(1).values - 2e-6).all()
    rows = torch.bincount(r.expert_idx.flatten().long(), minlength=n) * L
    assert torch.equal(r.expert_offsets.long().diff(), (rows + 127) // 128 * 128)


def test_every_launch_of_a_call_is_counted():
    """Scores of more samples than a grid dimension holds: two launches."""
    import paper_2503_02495_b200 as uoe
    prob = uoe.Problem(B=65541, L=33, L_valid=33, d=16, n=4, k=2, m=1, c=1, dtype="bf16")
    before = uoe.uoe_launch_count()
    uoe.uoe_route(prob, torch.zeros(prob.B, 33, 16, dtype=torch.bfloat16, device="cuda"), torch.zeros(16, 4, dtype=torch.bfloat16, device="cuda"))
    assert uoe.uoe_launch_count() - before == 2


# weight gradients cut into equal pieces over the SMs: ragged column tiles, 8-row slabs, one expert whose tiles are cut into
# many pieces, experts without rows, routed copies, and the pass without gates (the cut tiles added by their own launch)
def _bwd(**kw):
    base = dict(B=3, L=96, L_valid=96, m=6, c=3, d=128, n=4, k=2, d_ff=512, H=4, d_h=64, dtype="bf16", w_std=0.05)
    base.update(kw)
    return gen.tiny(**base)


WGRAD_CASES = {
    "ragged_columns_patch8": (_bwd(B=5, L=64, L_valid=61, m=8, c=5, d=640, n=3, k=2, d_ff=3 * 128, H=9), True),
    "one_expert_many_pieces": (_bwd(B=6, L=1024, L_valid=1000, m=8, c=8, d=128, n=1, k=1, d_ff=384, H=1), True),
    "experts_without_rows": (_bwd(B=2, n=12, k=1, d_ff=12 * 128, H=12), True),
    "routed_copies": (_bwd(B=4, L=140, L_valid=133, m=7, c=4, d=256, n=3, k=2, d_ff=3 * 256, H=6), True),
    "no_gates": (_bwd(B=7, L=256, L_valid=256, m=8, c=6, d=384, n=2, k=2, d_ff=2 * 256, H=2), False),
}


@pytest.mark.parametrize("half", ["mlp", "att"])
@pytest.mark.parametrize("name", list(WGRAD_CASES))
def test_weight_gradients_cut_into_pieces(name, half):
    from tests.test_gpu_mlp_backward import _run as run_mlp
    from tests.test_gpu_smha_backward import _run as run_att
    w, use_gate = WGRAD_CASES[name]
    got, ref = (run_mlp(w, False, use_gate) if half == "mlp" else run_att(w, False, use_gate))[:2]
    for g, r in zip(got, ref[:len(got)]):
        if np.abs(r).max() > 0:
            assert rel_inf(g, r) <= TOL
        else:
            assert np.all(g == 0)


# float32 grouped GEMM: both tile shapes, ragged K and N, patches that do not tile 128 rows, biases, padding rows.  Tolerance:
# sums of at most 256 fp32 products, 2^-24 * sqrt(256) relative per output, 1e-5 of the largest value leaves ten times that.
F32_CASES = {
    "small_tiles": dict(B=3, m=5, L=65, L_valid=60, d=52, n=3, k=2, c=3, d_ff=3 * 28),
    "large_tiles": dict(B=40, m=10, L=170, L_valid=165, d=200, n=3, k=2, c=5, d_ff=3 * 132),
    "large_whole_samples": dict(B=48, m=2, L=128, L_valid=128, d=256, n=4, k=2, c=2, d_ff=4 * 256),
}


@pytest.mark.parametrize("name", list(F32_CASES))
def test_float32_experts_with_biases(name):
    import paper_2503_02495_b200 as uoe
    w = gen.tiny(H=0, act="gelu_tanh", w_std=0.1, **F32_CASES[name])
    x, Wr = gen.make_x(w), gen.make_router(w)
    W1, W2 = gen.make_mlp_weights(w)
    b1, b2 = gen.store(gen.normal(5, 1, (w.n, w.d_e), 0.3), "f32"), gen.store(gen.normal(5, 2, (w.n, w.d), 0.3), "f32")
    prob = problem_of(w, "mlp", residual=False)
    xd = to_dev(x)
    r = uoe.uoe_route(prob, xd, to_dev(Wr))
    y = uoe.uoe_mlp_forward(prob, xd, to_dev(W1), to_dev(W2), r, b1=to_dev(b1), b2=to_dev(b2))
    ro = orc.with_selection(x.f64, Wr.f64, r.expert_idx.cpu().numpy(), r.patch_idx.cpu().numpy(), w.m, w.L_valid)
    ref = orc.mlp_forward(x.f64, W1.f64, W2.f64, ro, w.act, residual=False, b1=b1.f64, b2=b2.f64)
    assert rel_inf(to_f64(y), ref) <= 1e-5


# attention backward: one tile (at most 128 tokens per pair), its edge, and blocks of 64 streamed past tiles of 128
@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("l_p,c,L_valid", [(16, 8, 160), (8, 17, 260), (16, 4, 157), (32, 6, 250), (64, 5, 400), (1, 33, 40)],
                         ids=lambda v: str(v))
def test_attention_backward_tiles(l_p, c, L_valid, causal):
    from tests.test_gpu_smha_backward import _run as run_att
    m = max(c, -(-L_valid // l_p)) + 1
    w = gen.tiny(B=3, L=m * l_p, L_valid=min(L_valid, m * l_p), m=m, c=c, d=128, n=3, k=2, d_ff=0, H=6, d_h=64, dtype="bf16",
                 w_std=0.08, causal=causal)
    got, ref = run_att(w, False)
    for g, r in zip(got, ref[:len(got)]):
        assert rel_inf(g, r) <= TOL


# more tokens than 2^31: 32768 + 40 samples of 65536 rows of 16 bytes (34 GB in, 34 GB out); the last samples are past the limit
def _two_to_the_31(dtype):
    import paper_2503_02495_b200 as uoe
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 100 << 30:
        pytest.skip("needs 100 GB of device memory")
    f32 = dtype == "f32"
    prob = uoe.Problem(B=32768 + 40, L=65536, L_valid=65536, d=4 if f32 else 8, n=1, k=1, m=1024, c=1, d_e=4 if f32 else 0,
                       dtype=dtype, gate=False, residual=False, act="identity")
    x = torch.zeros(prob.B, prob.L, prob.d, dtype=prob.torch_dtype, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(2)
    for b in (0, prob.B - 1):
        x[b] = torch.randn(prob.L, prob.d, device="cuda", generator=g).to(prob.torch_dtype)
    return uoe, prob, x, g


def test_float32_rows_past_two_to_the_31():
    """1e-6 of the largest value: sums of four float32 products, twice."""
    uoe, prob, x, g = _two_to_the_31("f32")
    W1, W2 = (torch.randn(1, 4, 4, device="cuda", generator=g) for _ in range(2))
    patch = torch.randint(prob.m, (prob.B, 1, 1), device="cuda", generator=g).to(torch.int32)
    rows = prob.B * prob.l_p
    r = uoe.Routing(torch.zeros(prob.B, 1, dtype=torch.int32, device="cuda"), patch, torch.ones(prob.B, 1, 1, device="cuda"), None, None,
                    torch.tensor([0, (rows + 127) // 128 * 128], dtype=torch.int32, device="cuda"))
    y = uoe.uoe_mlp_forward(prob, x, W1, W2, r)
    for b in (0, prob.B - 1):
        t = int(patch[b]) * prob.l_p + torch.arange(prob.l_p, device="cuda")
        ref = torch.zeros(prob.L, prob.d, dtype=torch.float64, device="cuda")
        ref[t] = x[b, t].double() @ W1[0].double() @ W2[0].double()
        assert (y[b].double() - ref).abs().max() <= 1e-6 * ref.abs().max()


def test_router_gradient_of_rows_past_two_to_the_31():
    """With one expert the balance loss has no gradient, so the gate is given: two experts, p and 1 - p of every patch.  dW_r is a
    float32 sum over the last sample's 65536 rows, 2^-24 * sqrt(65536) relative; 1e-3 of the largest value."""
    uoe, prob, x, g = _two_to_the_31("bf16")
    prob.n = 2
    p = torch.full((prob.B, 2, prob.m), 0.5, device="cuda")
    p[:, 0] = 0.75
    p[:, 1] = 0.25
    dloss = torch.zeros(prob.B, device="cuda")
    dloss[-1] = 1.0
    dx, dWr = uoe.uoe_route_balance_backward(prob, x, torch.zeros(prob.d, 2, dtype=torch.bfloat16, device="cuda"), p, 1.0, dloss)
    # every patch goes to expert 0: f = (2, 0), dL/dg = f / m, the softmax Jacobian leaves +-0.75 * 0.25 * 2 / m, per token / l_p
    ref = x[-1].double().sum(0) * (0.75 * 0.25 * 2 / prob.m / prob.l_p)
    assert (dWr[:, 0].double() - ref).abs().max() <= 1e-3 * ref.abs().max()
    assert (dWr[:, 1].double() + ref).abs().max() <= 1e-3 * ref.abs().max()
    assert (dx[-1] == 0).all()


# whole tiles (many of them, operands past L2): 128 x 256 gathered and from copies, 128 x 128 beside 128 x 256, experts without rows
WHOLE_CASES = {
    "gathered_256": dict(B=34, L=512, l_p=32, d=1024, n=16, k=4, c=8, d_e=512),
    "copies_256": dict(B=24, L=480, l_p=24, d=1024, n=16, k=4, c=12, d_e=512),
    "gathered_128": dict(B=72, L=512, l_p=64, d=896, n=12, k=2, c=3, d_e=1024),
    "some_experts_idle": dict(B=48, L=512, l_p=16, d=1280, n=16, k=3, c=10, d_e=640, used=(0, 5, 6, 11, 15)),
}


@pytest.mark.parametrize("name", list(WHOLE_CASES))
def test_weight_gradients_of_whole_tiles(name):
    """Against float64 on the GPU with the identity as activation; the bfloat16 tolerance of the other gradients."""
    import paper_2503_02495_b200 as uoe
    kw = dict(WHOLE_CASES[name])
    used, l_p = kw.pop("used", None), kw.pop("l_p")
    p = uoe.Problem(**kw, m=kw["L"] // l_p, L_valid=kw["L"] - 5, act="identity", residual=False)
    g = torch.Generator(device="cuda").manual_seed(4)
    rn = lambda *s, std=1.0: (std * torch.randn(*s, device="cuda", generator=g)).bfloat16()
    x, dy, Wr = rn(p.B, p.L, p.d), rn(p.B, p.L, p.d), rn(p.d, p.n, std=0.05)
    x[:, p.L_valid:] = 0
    W1, W2 = rn(p.n, p.d, p.d_e, std=0.03), rn(p.n, p.d_e, p.d, std=0.03)
    r = uoe.uoe_route(p, x, Wr)
    if used:       # the same patches, the experts drawn from a few
        pick = torch.stack([torch.tensor(used, device="cuda")[torch.randperm(len(used), device="cuda", generator=g)[:p.k]].sort().values for _ in range(p.B)])
        r.expert_idx = pick.to(torch.int32)
        rows = torch.bincount(pick.flatten(), minlength=p.n) * p.l_a
        r.expert_offsets = torch.cat([rows.new_zeros(1), ((rows + 127) // 128 * 128).cumsum(0)]).to(torch.int32)
    sh = uoe.alloc_saved_h(p)
    uoe.uoe_mlp_forward(p, x, W1, W2, r, saved_h=sh)
    uoe.uoe_profile_enable(True)
    _, dW1, dW2, _ = uoe.uoe_mlp_backward(p, x, W1, W2, Wr, r, sh, dy)
    uoe.uoe_profile_enable(False)
    assert {"wgrad_W1", "wgrad_W2"} <= {label for label, _ in uoe.uoe_profile_records()}      # this case is one of whole tiles
    tok = (r.patch_idx.long()[..., None] * l_p + torch.arange(l_p, device="cuda")).flatten(2)          # [B, k, l_a]
    w = (r.gate.double().repeat_interleave(l_p, 2) * (tok < p.L_valid)).flatten(1)
    for e in range(p.n):
        b, s = (r.expert_idx == e).nonzero(as_tuple=True)
        xe = x.double()[b[:, None], tok[b, s]].flatten(0, 1)
        de = (dy.double()[b[:, None], tok[b, s]] * w.view(p.B, p.k, -1)[b, s][..., None]).flatten(0, 1)
        for got, ref in ((dW1[e], xe.T @ (de @ W2[e].double().T)), (dW2[e], (xe @ W1[e].double()).T @ de)):
            if len(b):
                assert (got.double() - ref).abs().max() <= TOL * ref.abs().max()
            else:
                assert (got == 0).all()


# one or two K blocks: whole lines per store of the forward epilogue, every tile width, CTA pairs, side-by-side projections
@pytest.mark.parametrize("d,d_e,B", [(64, 64, 3), (128, 320, 3), (64, 1152, 5), (128, 512, 3), (128, 1280, 260)])
def test_forward_of_short_contractions(d, d_e, B):
    """The pre-activation and y against float64 on the GPU, the bfloat16 tolerance of the other outputs."""
    import paper_2503_02495_b200 as uoe
    p = uoe.Problem(B=B, L=256, L_valid=250, d=d, n=3, k=2, m=4, c=3, d_e=d_e, residual=False)
    g = torch.Generator(device="cuda").manual_seed(6)
    rn = lambda *s, std=1.0: (std * torch.randn(*s, device="cuda", generator=g)).bfloat16()
    x, Wr, W1, W2 = rn(p.B, p.L, d), rn(d, p.n, std=0.1), rn(p.n, d, d_e, std=0.1), rn(p.n, d_e, d, std=0.1)
    b1, b2 = rn(p.n, d_e), rn(p.n, d)
    x[:, p.L_valid:] = 0
    r = uoe.uoe_route(p, x, Wr)
    sh = uoe.alloc_saved_h(p)
    y = uoe.uoe_mlp_forward(p, x, W1, W2, r, b1=b1, b2=b2, saved_h=sh)
    tok = (r.patch_idx.long()[..., None] * p.l_p + torch.arange(p.l_p, device="cuda")).flatten(2)
    ref = torch.zeros(p.B, p.L, d, dtype=torch.float64, device="cuda")
    for e in range(p.n):
        b, s = (r.expert_idx == e).nonzero(as_tuple=True)
        h = x.double()[b[:, None], tok[b, s]] @ W1[e].double() + b1[e].double()
        off = int(r.expert_offsets[e])
        assert (sh[off:off + h.shape[0] * p.l_a].double() - h.flatten(0, 1)).abs().max() <= TOL * h.abs().max()
        z = (torch.nn.functional.silu(h) @ W2[e].double() + b2[e].double()) * r.gate.double()[b, s].repeat_interleave(p.l_p, 1)[..., None]
        ref.index_put_((b[:, None].expand(-1, p.l_a), tok[b, s]), z * (tok[b, s] < p.L_valid)[..., None], accumulate=True)
    assert (y.double() - ref).abs().max() <= TOL * ref.abs().max()


@pytest.mark.parametrize("d,heads", [(64, 1), (128, 1), (640, 1), (1088, 2), (1280, 1)])
def test_attention_projections_of_short_contractions(d, heads):
    import paper_2503_02495_b200 as uoe
    w = gen.tiny(B=3, L=96, L_valid=90, m=6, c=4, d=d, n=2, k=2, d_ff=0, H=2 * heads, d_h=64, dtype="bf16", w_std=0.05, causal=True)
    x, Wr, ws = gen.make_x(w), gen.make_router(w, "att"), gen.make_attn_weights(w)
    prob = problem_of(w, "att", residual=False)
    r = uoe.uoe_route(prob, to_dev(x), to_dev(Wr))
    y = uoe.uoe_smha_forward(prob, to_dev(x), *(to_dev(q) for q in ws), r)
    ro = orc.with_selection(x.f64, Wr.f64, r.expert_idx.cpu().numpy(), r.patch_idx.cpu().numpy(), w.m, w.L_valid)
    ref = orc.smha_forward(x.f64, *[q.f64 for q in ws], ro, w.d_h, w.causal, residual=False)
    assert rel_inf(to_f64(y), ref) <= TOL


@pytest.mark.parametrize("heads", [1, 3])
def test_attention_of_pairs_with_fewer_key_tiles_than_others(heads):
    """Pairs that hold the last, nearly empty patch have one key tile less; more units than two per SM."""
    import paper_2503_02495_b200 as uoe
    w = gen.tiny(B=60 // heads, L=6 * 48, L_valid=5 * 48 + 1, m=6, c=3, d=64, n=3, k=3, d_ff=0, H=3 * heads, d_h=64, dtype="bf16", w_std=0.08)
    x, Wr = gen.make_x(w), gen.store(gen.make_router(w, "att").f64 * 20, w.dtype)
    ws = gen.make_attn_weights(w)
    prob = problem_of(w, "att", residual=False)
    r = uoe.uoe_route(prob, to_dev(x), to_dev(Wr))
    has_last = (r.patch_idx == w.m - 1).any(2)
    assert has_last.any() and not has_last.all()
    y = uoe.uoe_smha_forward(prob, to_dev(x), *(to_dev(q) for q in ws), r)
    ro = orc.with_selection(x.f64, Wr.f64, r.expert_idx.cpu().numpy(), r.patch_idx.cpu().numpy(), w.m, w.L_valid)
    assert rel_inf(to_f64(y), orc.smha_forward(x.f64, *[q.f64 for q in ws], ro, w.d_h, w.causal, residual=False)) <= TOL


# the combine's units of 64 vectors: slabs shorter than a unit, a vector longer, and of many; one to five slots per patch (two
# are in flight), whole samples per expert, padding rows, more units than warps
@pytest.mark.parametrize("kw", [dict(B=2, L=9, L_valid=8, m=9, c=7, d=4, n=6, k=5, d_ff=24), dict(B=3, L=13 * 6, L_valid=70, m=6, c=4, d=20, n=3, k=3, d_ff=12),
                                dict(B=2, L=64, L_valid=50, m=2, c=2, d=260, n=5, k=4, d_ff=40), dict(B=40, L=1024, L_valid=1000, m=16, c=9, d=128, n=3, k=1, d_ff=12)],
                         ids=["short_slabs", "a_vector_over", "whole_samples", "many_units"])
def test_combine_of_slabs(kw):
    """float32: sums of at most 260 products per layer, 1e-4 of the largest value as for the other float32 results."""
    import paper_2503_02495_b200 as uoe
    w = gen.tiny(**kw)
    x, Wr = gen.make_x(w), gen.make_router(w)
    W1, W2 = gen.make_mlp_weights(w)
    prob = problem_of(w, "mlp")
    r = uoe.uoe_route(prob, to_dev(x), to_dev(Wr))
    y = to_f64(uoe.uoe_mlp_forward(prob, to_dev(x), to_dev(W1), to_dev(W2), r))
    ro = orc.with_selection(x.f64, Wr.f64, r.expert_idx.cpu().numpy(), r.patch_idx.cpu().numpy(), w.m, w.L_valid)
    assert rel_inf(y, orc.mlp_forward(x.f64, W1.f64, W2.f64, ro, w.act, residual=True)) <= 1e-4


# projections and attention in one kernel: one tile (short, padded, eight-row patches, full) and clusters of two to eight tiles
# (real keys that end before the pair's last tile, causal, rotary)
FUSED_CASES = {
    "short": (_att(B=3, L=96, L_valid=96, m=6, c=3, d=128, n=4, k=2, H=4), 0),
    "causal_pad_rope": (_att(B=5, L=128, L_valid=121, m=8, c=7, d=128, n=3, k=2, H=3, causal=True), 32),
    "patch8": (_att(B=4, L=96, L_valid=90, m=12, c=9, d=384, n=4, k=2, H=4), 0),
    "one_full_tile": (_att(B=4, L=256, L_valid=256, m=8, c=4, d=512, n=4, k=2, H=4), 0),
    "two_tiles_causal": (_att(B=4, L=512, L_valid=500, m=16, c=8, d=512, n=4, k=2, H=4, causal=True), 0),
    "three_tiles_no_real_key_in_the_last": (_att(B=2, L=768, L_valid=400, m=6, c=3, d=128, n=4, k=2, H=4), 0),
    "eight_tiles": (_att(B=2, L=2048, L_valid=2048, m=32, c=16, d=256, n=4, k=2, H=4), 0),
    "whole_samples_causal_rope": (_att(B=1, L=1024, L_valid=1000, m=16, c=16, d=128, n=4, k=2, H=4, causal=True), 64),
}


@pytest.mark.parametrize("name", list(FUSED_CASES))
def test_projection_and_attention_in_one_kernel(name):
    import paper_2503_02495_b200 as uoe
    w, d_rope = FUSED_CASES[name]
    x, Wr = gen.make_x(w), gen.store(gen.make_router(w, "att").f64 * 20, w.dtype)
    ws = gen.make_attn_weights(w)
    prob = problem_of(w, "att", residual=False, d_rope=d_rope)
    xd, Wrd, wd = to_dev(x), to_dev(Wr), [to_dev(q) for q in ws]
    r = uoe.uoe_route(prob, xd, Wrd)
    dy = gen.make_dy(w)
    uoe.uoe_profile_enable(True)
    y = uoe.uoe_smha_forward(prob, xd, *wd, r)
    got = uoe.uoe_smha_backward(prob, xd, *wd, Wrd, r, to_dev(dy))
    torch.cuda.synchronize()
    uoe.uoe_profile_enable(False)
    assert [n for n, _ in uoe.uoe_profile_records()].count("smha_fused") == 2
    ro = orc.with_selection(x.f64, Wr.f64, r.expert_idx.cpu().numpy(), r.patch_idx.cpu().numpy(), w.m, w.L_valid)
    ref_y = orc.smha_forward(x.f64, *[q.f64 for q in ws], ro, w.d_h, w.causal, residual=False, d_rope=d_rope)
    assert rel_inf(to_f64(y), ref_y) <= TOL
    ref = orc.smha_backward(x.f64, *[q.f64 for q in ws], Wr.f64, ro, dy.f64, w.d_h, w.causal, residual=False, d_rope=d_rope)
    for g, f in zip(got, ref[:6]):
        assert rel_inf(to_f64(g), f) <= TOL


# which calls take that kernel, on both sides of each line (pairs against SMs, tokens per pair, whole tiles, resident clusters, width), and
# widths whose last chunk of output columns is half a chunk; a width that 128 does not divide has no backward.  Pairs are counted in
# SMs: (twice the SMs, + 2) and so on, two experts per sample.
def _pairs(times, more=0):
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 148
    return (times * sms + more) // 2


def _short(pairs, l_a, **kw):
    return _att(**{**dict(B=pairs, L=2 * l_a, L_valid=2 * l_a, m=4, c=2, d=128, n=4, k=2, H=4), **kw})


DISPATCH = {
    "d192_one_tile": (lambda: _att(B=3, L=192, L_valid=185, m=6, c=3, d=192, n=4, k=2, H=4), True, None),
    "d448_one_tile": (lambda: _att(B=3, L=192, L_valid=185, m=6, c=3, d=448, n=4, k=2, H=4, causal=True), True, None),
    "d192_cluster": (lambda: _att(B=3, L=512, L_valid=500, m=16, c=8, d=192, n=4, k=2, H=4, causal=True), True, None),
    "d448_cluster": (lambda: _att(B=2, L=768, L_valid=700, m=12, c=6, d=448, n=4, k=2, H=4), True, None),
    "d512": (lambda: _short(4, 64, d=512), True, True),
    "d640": (lambda: _short(4, 64, d=640), False, True),
    "two_pairs_per_sm": (lambda: _short(_pairs(2), 16), True, True),
    "more_pairs_short": (lambda: _short(_pairs(2, 2), 16), True, False),
    "four_pairs_per_sm": (lambda: _short(_pairs(4), 32), True, False),
    "many_pairs_32": (lambda: _short(_pairs(4, 2), 32), False, False),
    "many_pairs_48": (lambda: _short(_pairs(4, 2), 48, L=96, m=6, c=3), True, False),
    "many_pairs_96": (lambda: _short(_pairs(5, 2), 96, L=192, L_valid=180, m=12, c=6), True, True),
    "many_pairs_128": (lambda: _short(_pairs(5, 2), 128, causal=True), True, True),
    "ragged_tiles": (lambda: _att(B=4, L=320, L_valid=320, m=10, c=5, d=128, n=4, k=2, H=4), False, False),
    "nine_tiles": (lambda: _att(B=1, L=2304, L_valid=2300, m=18, c=9, d=128, n=2, k=1, H=2), False, False),
    "clusters_beyond_a_wave": (lambda: _short(_pairs(1), 256, m=16, c=8), False, False),
}


@pytest.mark.parametrize("name", list(DISPATCH))
def test_which_calls_take_the_one_kernel(name):
    import paper_2503_02495_b200 as uoe
    make, forward, backward = DISPATCH[name]
    w = make()
    x, Wr = gen.make_x(w), gen.store(gen.make_router(w, "att").f64 * 20, w.dtype)
    ws, dy = gen.make_attn_weights(w), gen.make_dy(w)
    prob = problem_of(w, "att", residual=False)
    xd, Wrd, wd = to_dev(x), to_dev(Wr), [to_dev(q) for q in ws]
    r = uoe.uoe_route(prob, xd, Wrd)
    ro = orc.with_selection(x.f64, Wr.f64, r.expert_idx.cpu().numpy(), r.patch_idx.cpu().numpy(), w.m, w.L_valid)
    fs = [q.f64 for q in ws]

    def launched(call):
        uoe.uoe_profile_enable(True)
        out = call()
        torch.cuda.synchronize()
        uoe.uoe_profile_enable(False)
        return out, "smha_fused" in [n for n, _ in uoe.uoe_profile_records()]

    y, fused = launched(lambda: uoe.uoe_smha_forward(prob, xd, *wd, r))
    assert fused == forward
    assert rel_inf(to_f64(y), orc.smha_forward(x.f64, *fs, ro, w.d_h, w.causal, residual=False)) <= TOL
    if backward is None:
        return
    got, fused = launched(lambda: uoe.uoe_smha_backward(prob, xd, *wd, Wrd, r, to_dev(dy)))
    assert fused == backward
    for g, f in zip(got, orc.smha_backward(x.f64, *fs, Wr.f64, ro, dy.f64, w.d_h, w.causal, residual=False)[:6]):
        assert rel_inf(to_f64(g), f) <= TOL
