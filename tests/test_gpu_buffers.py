"""What the library asks of a caller's buffers, and no more: workspaces and saved arrays that are multiples of 16 bytes but not
of 32, rows of lse that hold no key.  References: the float64 oracle on the GPU's own selection (bfloat16: 2e-2 of the largest
value, as in the other parity tests) and the same call on buffers of the allocator, bit for bit.
"""
import pytest
import torch

import uoe_inputs as gen
from oracle import uoe_oracle as orc
from tests.helpers import problem_of, rel_inf, to_dev, to_f64

pytestmark = pytest.mark.gpu

TOL = 2e-2


def _w(**kw):
    base = dict(B=4, L=256, L_valid=256, m=8, c=4, d=128, n=4, k=2, d_ff=0, H=4, d_h=64, dtype="bf16", w_std=0.08, causal=False)
    base.update(kw)
    return gen.tiny(**base)


def _at_16(nbytes):
    """nbytes of device memory at 16 modulo 32, full of NaN patterns."""
    buf = torch.full((nbytes + 32,), 255, dtype=torch.uint8, device="cuda")
    ws = buf[16:16 + nbytes]
    assert ws.data_ptr() % 32 == 16
    return ws


def _ws(nbytes, at_16=True):
    from paper_2503_02495_b200 import binding as B
    ws = _at_16(nbytes) if at_16 else torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    B._check(B._lib.uoe_workspace_init(B._ptr(ws), nbytes, B._stream()), "uoe_workspace_init")
    return ws


# every kernel of the attention half that writes a routed buffer: projections and attention in one kernel (one tile per pair, a
# cluster), one CTA per unit and two pipelines per CTA with the output projection as a launch of its own
ATT = {
    "one_tile": _w(d=512),
    "cluster_causal": _w(L=512, L_valid=500, m=16, c=8, d=256, causal=True),
    "two_heads": _w(L=192, L_valid=185, m=6, c=4, d=128, H=8),
    "two_heads_many_units": _w(B=80, L_valid=250, c=6, n=2, H=4),
}


@pytest.mark.parametrize("name", list(ATT))
def test_attention_on_a_workspace_of_16_bytes(name):
    import paper_2503_02495_b200 as uoe
    w = ATT[name]
    x, Wr, ws, dy = gen.make_x(w), gen.store(gen.make_router(w, "att").f64 * 20, w.dtype), gen.make_attn_weights(w), gen.make_dy(w)
    prob = problem_of(w, "att", residual=False)
    xd, Wrd, wd, dyd = to_dev(x), to_dev(Wr), [to_dev(q) for q in ws], to_dev(dy)
    r = uoe.uoe_route(prob, xd, Wrd)
    y = uoe.uoe_smha_forward(prob, xd, *wd, r, ws=_ws(uoe.uoe_workspace_bytes(prob, uoe.UOE_OP_SMHA_FWD)))
    got = uoe.uoe_smha_backward(prob, xd, *wd, Wrd, r, dyd, ws=_ws(uoe.uoe_workspace_bytes(prob, uoe.UOE_OP_SMHA_BWD)))
    ro = orc.with_selection(x.f64, Wr.f64, r.expert_idx.cpu().numpy(), r.patch_idx.cpu().numpy(), w.m, w.L_valid)
    fs = [q.f64 for q in ws]
    assert rel_inf(to_f64(y), orc.smha_forward(x.f64, *fs, ro, w.d_h, w.causal, residual=False)) <= TOL
    for g, f in zip(got, orc.smha_backward(x.f64, *fs, Wr.f64, ro, dy.f64, w.d_h, w.causal, residual=False)[:6]):
        assert rel_inf(to_f64(g), f) <= TOL
    assert torch.equal(y, uoe.uoe_smha_forward(prob, xd, *wd, r))
    for g, f in zip(got, uoe.uoe_smha_backward(prob, xd, *wd, Wrd, r, dyd)):
        assert torch.equal(g, f)


@pytest.mark.parametrize("kw", [dict(d=512, d_ff=4 * 256), dict(d=256, d_ff=4 * 384, H=8, L=320, L_valid=301, m=5, c=3)],
                         ids=["narrow_experts", "two_layers_ragged"])
def test_block_and_mlp_on_buffers_of_16_bytes(kw):
    import paper_2503_02495_b200 as uoe
    w = _w(**kw)
    x, dy = gen.make_x(w), to_dev(gen.make_dy(w))
    h = dict(zip(("Wq", "Wk", "Wv", "Wo", "W1", "W2"), gen.make_attn_weights(w) + gen.make_mlp_weights(w)),
             Wr_att=gen.make_router(w, "att"), Wr_mlp=gen.make_router(w, "mlp"))
    wd = {q: to_dev(v) for q, v in h.items()}
    pa, pm, xd = problem_of(w, "att"), problem_of(w, "mlp"), to_dev(x)

    def run(ws_of, saved):
        ra, rm, u = uoe.alloc_routing(pa), uoe.alloc_routing(pm), torch.empty_like(xd)
        y = uoe.uoe_block_forward(pa, pm, xd, wd, r_att=ra, r_mlp=rm, u=u, saved_h=saved, ws=ws_of(uoe.uoe_block_workspace_bytes(pa, pm)))
        g = uoe.uoe_mlp_backward(pm, u, wd["W1"], wd["W2"], wd["Wr_mlp"], rm, saved, dy, ws=ws_of(uoe.uoe_workspace_bytes(pm, uoe.UOE_OP_MLP_BWD)))
        y2 = uoe.uoe_mlp_forward(pm, u, wd["W1"], wd["W2"], rm, saved_h=saved, ws=ws_of(uoe.uoe_workspace_bytes(pm, uoe.UOE_OP_MLP_FWD)))
        return [u, y, y2, *g], ra, rm

    size = (uoe.uoe_max_routed_rows(pm), w.d_e)
    got, ra, rm = run(_ws, _at_16(size[0] * size[1] * 2).view(torch.bfloat16).view(size))
    sel = lambda r, src, W: orc.with_selection(src, W.f64, r.expert_idx.cpu().numpy(), r.patch_idx.cpu().numpy(), w.m, w.L_valid)
    u64 = to_f64(got[0])
    assert rel_inf(u64, orc.smha_forward(x.f64, *[h[q].f64 for q in ("Wq", "Wk", "Wv", "Wo")], sel(ra, x.f64, h["Wr_att"]), w.d_h, w.causal)) <= TOL
    assert rel_inf(to_f64(got[1]), orc.mlp_forward(u64, h["W1"].f64, h["W2"].f64, sel(rm, u64, h["Wr_mlp"]), w.act)) <= TOL
    ref, _, _ = run(lambda nbytes: _ws(nbytes, at_16=False), torch.zeros(size, dtype=torch.bfloat16, device="cuda"))
    for g, f in zip(got, ref):
        assert torch.equal(g, f)
