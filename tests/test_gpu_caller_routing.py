"""Routing arrays a caller builds: an expert named twice by a sample, an index out of range, pairs whose slots are all unused.
References: the float64 oracle on the same arrays; tolerances as in the other parity tests (1e-4 and 2e-2 of the largest value)."""
import numpy as np
import pytest
import torch

import uoe_inputs as gen
from oracle import uoe_oracle as orc
from tests.helpers import problem_of, rel_inf, to_dev, to_f64

pytestmark = pytest.mark.gpu


def _mlp(**kw):
    base = dict(B=4, L=120, L_valid=113, m=6, c=3, d=16, n=3, k=2, d_ff=3 * 16, H=0, dtype="f32")
    return gen.tiny(**{**base, **kw})


def _att(**kw):
    base = dict(B=4, L=120, L_valid=113, m=6, c=3, d=128, n=3, k=2, d_ff=0, H=3, d_h=64, dtype="bf16", w_std=0.08)
    return gen.tiny(**{**base, **kw})


class Layer:
    """One half of a block with its inputs and the router's own arrays, which the tests change."""

    def __init__(self, w, half, d_rope=0):
        import paper_2503_02495_b200 as uoe
        self.uoe, self.w, self.half, self.d_rope = uoe, w, half, d_rope
        self.x, self.Wr = gen.make_x(w), gen.store(gen.make_router(w, half).f64 * 20, w.dtype)
        self.ws = gen.make_mlp_weights(w) if half == "mlp" else gen.make_attn_weights(w)
        self.prob = problem_of(w, half, residual=False, d_rope=d_rope)
        self.xd, self.Wrd, self.wd = to_dev(self.x), to_dev(self.Wr), [to_dev(q) for q in self.ws]
        self.r = uoe.uoe_route(self.prob, self.xd, self.Wrd)

    def use(self, expert_idx, patch_idx):
        """Takes these arrays, with gates and offsets that belong to them; returns the oracle's routing."""
        ro = orc.with_selection(self.x.f64, self.Wr.f64, expert_idx, patch_idx, self.w.m, self.w.L_valid)
        dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a)).to(device="cuda", dtype=t)
        self.r.expert_idx, self.r.patch_idx = dev(expert_idx, torch.int32), dev(patch_idx, torch.int32)
        self.r.gate, self.r.expert_offsets = dev(ro.gate, torch.float32), dev(ro.offsets, torch.int32)
        return ro

    def forward(self):
        f = self.uoe.uoe_mlp_forward if self.half == "mlp" else self.uoe.uoe_smha_forward
        return f(self.prob, self.xd, *self.wd, self.r)

    def backward(self, dy):
        saved = [torch.zeros(self.uoe.uoe_max_routed_rows(self.prob), self.w.d_e, dtype=torch.bfloat16, device="cuda")] if self.half == "mlp" else []
        f = self.uoe.uoe_mlp_backward if self.half == "mlp" else self.uoe.uoe_smha_backward
        return f(self.prob, self.xd, *self.wd, self.Wrd, self.r, *saved, to_dev(dy))

    def reference(self, ro):
        fs = [q.f64 for q in self.ws]
        if self.half == "mlp":
            return orc.mlp_forward(self.x.f64, *fs, ro, self.w.act, residual=False)
        return orc.smha_forward(self.x.f64, *fs, ro, self.w.d_h, self.w.causal, residual=False, d_rope=self.d_rope)


# both sides of the sample count from which the rows of the pairs come from a kernel of their own
@pytest.mark.parametrize("B", [4, 530])
@pytest.mark.parametrize("half", ["mlp", "att"])
def test_expert_named_twice_adds_both_contributions(half, B):
    """More pairs name an expert than there are samples: the place of a pair in its expert's region exceeds B."""
    w = _mlp(B=B) if half == "mlp" else _att(B=B, L=40, L_valid=37, m=2, c=1)
    layer = Layer(w, half, d_rope=32 if half == "att" else 0)
    patch = layer.r.patch_idx.cpu().numpy().copy()
    patch[:, 1] = patch[:, 0]
    ro = layer.use(np.full((w.B, w.k), w.n - 1, dtype=np.int32), patch)
    assert rel_inf(to_f64(layer.forward()), layer.reference(ro)) <= (1e-4 if half == "mlp" else 2e-2)


@pytest.mark.parametrize("bad", [-1, 3, 1 << 20])
@pytest.mark.parametrize("B", [4, 530])
@pytest.mark.parametrize("half", ["mlp", "att"])
def test_expert_out_of_range_is_reported(half, B, bad):
    """The call returns the status code; samples in front of the bad one are what they are without it."""
    w = _mlp(B=B) if half == "mlp" else _att(B=B, L=40, L_valid=37, m=2, c=1)
    layer = Layer(w, half, d_rope=32 if half == "att" else 0)
    good = layer.forward()
    layer.r.expert_idx[-1, 0] = bad
    y = torch.zeros_like(good)
    f = layer.uoe.uoe_mlp_forward if half == "mlp" else layer.uoe.uoe_smha_forward
    with pytest.raises(layer.uoe.UoeError) as ei:
        f(layer.prob, layer.xd, *layer.wd, layer.r, y=y)
    assert ei.value.status == 6
    assert torch.equal(y[:-1], good[:-1])


@pytest.mark.parametrize("bad", [-1, 3])
@pytest.mark.parametrize("half", ["mlp", "att"])
def test_expert_out_of_range_is_reported_by_the_backward(half, bad):
    w = _att(B=5) if half == "att" else _mlp(B=5, d=128, d_ff=3 * 128, dtype="bf16")
    layer = Layer(w, half, d_rope=16 if half == "att" else 0)
    layer.r.expert_idx[2, 1] = bad
    with pytest.raises(layer.uoe.UoeError) as ei:
        layer.backward(gen.make_dy(w))
    assert ei.value.status == 6


# few units (a CTA each) and more units than SMs (two pipelines per SM), with the output projection inside the kernel and without
@pytest.mark.parametrize("heads", [1, 2])
@pytest.mark.parametrize("B", [12, 240])
def test_pairs_without_a_patch(B, heads):
    """Every third pair has only unused slots: no keys, no rows to add, no gradient; the others are not disturbed."""
    w = _att(B=B, L=48, L_valid=45, m=3, c=2, n=2, H=2 * heads)
    layer = Layer(w, "att")
    patch = layer.r.patch_idx.cpu().numpy().copy()
    patch.reshape(B * w.k, w.c)[::3] = -1
    ro = layer.use(layer.r.expert_idx.cpu().numpy(), patch)
    for _ in range(3):
        assert rel_inf(to_f64(layer.forward()), layer.reference(ro)) <= 2e-2
    dy = gen.make_dy(w)
    ref = orc.smha_backward(layer.x.f64, *[q.f64 for q in layer.ws], layer.Wr.f64, ro, dy.f64, w.d_h, w.causal, False)
    for g, r in zip(layer.backward(dy), ref):
        assert rel_inf(to_f64(g), r) <= 2e-2


# one routed row per (row, head): every kernel that produces lse -- one tile per pair and clusters in one kernel with the
# projections, a CTA per unit and two pipelines per CTA, each with the output projection inside and without
LSE = {
    "one_tile": dict(B=12, L=48, L_valid=45, m=3, c=2, n=2, H=2),
    "cluster": dict(B=4, L=512, L_valid=500, m=16, c=8, n=2, H=2, causal=True),
    "cta_per_unit_out": dict(B=6, L=320, L_valid=311, m=10, c=5, n=2, H=2),
    "cta_per_unit": dict(B=12, L=48, L_valid=45, m=3, c=2, n=2, H=4),
    "pipelines_out": dict(B=120, L=320, L_valid=311, m=10, c=5, n=2, H=2),
    "pipelines": dict(B=240, L=48, L_valid=45, m=3, c=2, n=2, H=4),
}


@pytest.mark.parametrize("name", list(LSE))
def test_log_sum_exp_of_every_routed_row(name):
    """Every third pair has only unused slots (-inf), every fifth one an unused last slot.  Scores of a few units, q and k rounded
    to bfloat16 (2^-9 each): 2e-2 of the largest log-sum-exp, as for the other bfloat16 results."""
    w = _att(**LSE[name])
    layer = Layer(w, "att")
    patch = layer.r.patch_idx.cpu().numpy().copy()
    flat = patch.reshape(w.B * w.k, w.c)
    flat[::5, -1] = -1
    flat[::3] = -1
    ro = layer.use(layer.r.expert_idx.cpu().numpy(), patch)
    heads = w.d_g // w.d_h
    lse = torch.full((layer.uoe.uoe_max_routed_rows(layer.prob), heads), 77.0, device="cuda")
    y = layer.uoe.uoe_smha_forward(layer.prob, layer.xd, *layer.wd, layer.r, lse=lse)
    ref_y, ref = orc.smha_forward(layer.x.f64, *[q.f64 for q in layer.ws], ro, w.d_h, w.causal, residual=False, return_lse=True)
    assert rel_inf(to_f64(y), ref_y) <= 2e-2
    got, top = to_f64(lse), max(np.abs(v).max() for v in ref.values())
    l_a = w.c * (w.L // w.m)
    for b in range(w.B):
        for s in range(w.k):
            row = orc.buffer_row(ro, b, s)
            for hd in range(heads):
                have = got[row:row + l_a, hd]
                if (b, s, hd) not in ref:
                    assert np.all(have == -np.inf)
                else:
                    want = ref[b, s, hd]
                    assert np.abs(have[:len(want)] - want).max() <= 2e-2 * top


@pytest.mark.parametrize("causal", [False, True])
def test_clusters_with_unused_slots_and_a_pair_without_a_patch(causal):
    """Pairs of two 128-row tiles in one kernel: fewer keys than tiles, none at all, an expert out of range."""
    w = _att(B=5, L=512, L_valid=500, m=16, c=8, n=3, k=2, H=3, causal=causal)
    layer = Layer(w, "att", d_rope=32)
    patch = layer.r.patch_idx.cpu().numpy().copy()
    flat = patch.reshape(w.B * w.k, w.c)
    flat[1, 1:] = -1
    flat[4, 4:] = -1
    flat[7] = -1
    ro = layer.use(layer.r.expert_idx.cpu().numpy(), patch)
    good = layer.forward()
    assert rel_inf(to_f64(good), layer.reference(ro)) <= 2e-2
    dy = gen.make_dy(w)
    ref = orc.smha_backward(layer.x.f64, *[q.f64 for q in layer.ws], layer.Wr.f64, ro, dy.f64, w.d_h, w.causal, False, d_rope=32)
    for g, r in zip(layer.backward(dy), ref):
        assert rel_inf(to_f64(g), r) <= 2e-2
    layer.r.expert_idx[-1, 0] = 1 << 20
    y = torch.zeros_like(good)
    with pytest.raises(layer.uoe.UoeError) as ei:
        layer.uoe.uoe_smha_forward(layer.prob, layer.xd, *layer.wd, layer.r, y=y)
    assert ei.value.status == 6
    assert torch.equal(y[:-1], good[:-1])
