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


# one pass over x for dW_r and dx: every column-block width, row segments (patches above 64 rows), one-row patches,
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
