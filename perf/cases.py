"""Workloads for timing the library: what programs that use a Union-of-Experts block have it do.

A case is a plain dict.  `kind` says which program it is:
  block_fwd    inference: UoEBlock.forward (router -> SMHA -> router -> UoME)
  block_train  a training step of a whole block: forward, UoME backward, SMHA backward
  mlp_train    a training step of a UoME layer alone (no attention half): forward and backward
  mlp_f32      float32 UoME forward through the per-half entry points, with biases
  router_train the router on its own with the load-balancing loss: routing with dynamic capacity, the loss and its
               gradient (a program that trains or probes the router of a layer)
The other keys are the sizes and options of the layer (the letters of uoe_problem; d_e is the hidden width of one MLP
expert, heads the attention heads of one expert, skew the logit by which every sample is pulled towards one expert).

listed() holds the cases, draw() makes more of the same ranges, prepare() makes what a program holds before the call,
run() is one pass through the public entry points, work() the bytes and operations a pass cannot do without, and
tolerance() how far two correct implementations of the same precision may be apart.
"""
from __future__ import annotations

import math

import torch

import paper_2503_02495_b200 as uoe
from paper_2503_02495_b200.block import UoEBlock

HEAD_DIM = 64          # the width of a head the attention kernels work with


def _case(kind, B, L_valid, l_p, d, n, k, m, c, d_e=0, heads=0, act="silu", causal=False, d_rope=0, skew=0.0, w_std=0.02):
    return {"kind": kind, "B": B, "L_valid": L_valid, "l_p": l_p, "d": d, "n": n, "k": k, "m": m, "c": c, "d_e": d_e,
            "heads": heads, "act": act, "causal": causal, "d_rope": d_rope, "skew": skew, "w_std": w_std}


def listed():
    lm = dict(L_valid=512, l_p=32, d=512, n=8, k=4, m=16, c=8, d_e=256, heads=1, causal=True)
    vit = dict(B=256, L_valid=197, l_p=16, d=384, n=6, k=3, m=14, c=7, d_e=256, heads=1)
    wide = dict(B=4, L_valid=2048, l_p=32, d=1024, n=8, k=4, m=64, c=32, d_e=512, heads=2, causal=True, d_rope=32)
    cases = {
        # one sequence through the language-model block: the latency of an interactive request
        "lm_one_sequence": _case("block_fwd", B=1, **lm),
        # the language-model block on a batch of sequences (scoring, prefill)
        "lm_forward": _case("block_fwd", B=16, **lm),
        # long documents, bidirectional attention: 64-token patches, a quarter of them per expert
        "long_forward": _case("block_fwd", B=8, L_valid=4096, l_p=64, d=256, n=4, k=2, m=64, c=16, d_e=256, heads=1),
        # image tokens: many short samples padded to whole patches
        "vit_forward": _case("block_fwd", **vit),
        # a wider language-model block: two heads per expert, 512-wide experts, rotary positions
        "wide_forward": _case("block_fwd", **wide),
        # sizes that fit no tile: 20-token patches, five experts, a ragged last patch, odd widths
        "ragged_forward": _case("block_fwd", B=6, L_valid=1003, l_p=20, d=320, n=5, k=2, m=51, c=17, d_e=192, heads=1),
        # training steps of the language-model, image and wide blocks (the wide one with unequal expert loads)
        "lm_train": _case("block_train", B=16, **lm),
        "vit_train": _case("block_train", **vit),
        "wide_train": _case("block_train", skew=0.5, **wide),
        # the MLP layer of a large language model: training step
        "scale_train": _case("mlp_train", B=8, L_valid=4096, l_p=128, d=4096, n=16, k=4, m=32, c=16, d_e=1024, w_std=0.01),
        # float32 layer with biases and the exact GELU (small models, numerics-sensitive use)
        "f32_forward": _case("mlp_f32", B=2, L_valid=256, l_p=32, d=256, n=4, k=2, m=8, c=4, d_e=256, act="gelu_erf"),
        # router training with the balance loss and dynamic capacity
        "router_train": _case("router_train", B=16, L_valid=2048, l_p=32, d=1024, n=16, k=4, m=64, c=32),
    }
    return [dict(case, name=name) for name, case in cases.items()]


# ---------------------------------------------------------------------------------------------------------------
# drawn cases
# ---------------------------------------------------------------------------------------------------------------

def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _rough_us(case):
    """A rough cost that keeps drawn cases below the largest listed one (rates well below what kernels reach)."""
    w = work(case)
    if case["kind"] == "mlp_f32":
        return w["flops"] / 4e6 + w["bytes"] / 1e6
    l_a = case["c"] * case["l_p"]
    attn = 4.0 * case["B"] * case["k"] * l_a * l_a * HEAD_DIM * case["heads"] * (3.5 if "train" in case["kind"] else 1.0)
    return max(0.0, w["flops"] - attn) / 300e6 + attn / 60e6 + w["bytes"] / 1e6


def _draw_once(rng):
    kind = rng.choice(["block_fwd"] * 6 + ["block_train"] * 3 + ["mlp_train", "mlp_f32", "router_train"])
    train = kind in ("block_train", "mlp_train")
    # patches: mostly lengths that divide a 128-row tile, sometimes any length
    l_p = rng.choice([16, 16, 32, 32, 64, 64, 128, 8, rng.randint(5, 80)])
    length = _log_int(rng, 96, 4096)
    m = max(2, min(96, round(length / l_p)))
    L = m * l_p
    L_valid = L - (rng.randrange(l_p) if rng.random() < 0.4 else 0)
    n = rng.choice([2, 4, 4, 6, 8, 8, 12, 16, rng.randint(2, 16)])
    k = max(1, min(n, round(n * rng.choice([0.25, 0.5, 0.5, 1.0]))))
    c = max(1, min(m, round(m * rng.uniform(0.2, 1.0))))
    B = _log_int(rng, 1, max(1, min(256, 65536 // L)))
    skew = rng.choice([0.0, 0.0, 0.5])
    if kind == "mlp_f32":
        return _case(kind, B, L_valid, l_p, 4 * _log_int(rng, 16, 128), n, k, m, c, d_e=4 * _log_int(rng, 16, 96),
                     act=rng.choice(["gelu_erf", "gelu_tanh", "silu"]), skew=skew)
    if kind == "router_train":
        return _case(kind, B, L_valid, l_p, 64 * _log_int(rng, 2, 32), n, k, m, c, skew=skew)
    if kind == "mlp_train":
        return _case(kind, B, L_valid, l_p, 128 * _log_int(rng, 4, 32), n, k, m, c, d_e=128 * _log_int(rng, 2, 8),
                     act=rng.choice(["silu", "silu", "gelu_tanh"]), skew=skew, w_std=0.01)
    step = 128 if train else 64
    return _case(kind, B, L_valid, l_p, step * _log_int(rng, 256 // step, 1024 // step), n, k, m, c,
                 d_e=rng.choice([256, 256, step * _log_int(rng, 1, 768 // step)]), heads=rng.choice([1, 1, 1, 2]),
                 act=rng.choice(["silu", "silu", "gelu_erf"]), causal=rng.random() < 0.5, d_rope=rng.choice([0, 0, 32, 64]),
                 skew=skew)


def draw(rng):
    while True:
        case = _draw_once(rng)
        if _rough_us(case) <= 2000.0:
            return case


# ---------------------------------------------------------------------------------------------------------------
# a program's state and one pass
# ---------------------------------------------------------------------------------------------------------------

def _problem(case, half):
    L = case["m"] * case["l_p"]
    return uoe.Problem(B=case["B"], L=L, L_valid=case["L_valid"], d=case["d"], n=case["n"], k=case["k"], m=case["m"], c=case["c"],
                       d_e=case["d_e"] if half == "mlp" else 0, H=case["n"] * case["heads"] if half == "att" else 0,
                       d_h=HEAD_DIM if half == "att" else 0, dtype="f32" if case["kind"] == "mlp_f32" else "bf16",
                       act=case["act"], causal=case["causal"] and half == "att", d_rope=case["d_rope"] if half == "att" else 0,
                       dynamic_c=case["kind"] == "router_train")


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    B, d, n, d_e, d_g = case["B"], case["d"], case["n"], case["d_e"], case["heads"] * HEAD_DIM
    L = case["m"] * case["l_p"]
    dtype = torch.float32 if case["kind"] == "mlp_f32" else torch.bfloat16

    def normal(*shape, std=1.0):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32).mul_(std).to(dtype)

    def tokens(shift=None):
        t = torch.randn(B, L, d, generator=gen, device="cuda", dtype=torch.float32)
        if shift is not None:
            t += shift[:, None, :]
        t[:, case["L_valid"]:] = 0                       # rows past the real tokens are zero
        return t.to(dtype)

    routers = {"Wr_att": normal(d, n, std=0.02), "Wr_mlp": normal(d, n, std=0.02)}
    shift = None
    if case["skew"] > 0:      # every sample leans towards one expert, popular experts more often (Zipf)
        pop = 1.0 / torch.arange(1, n + 1, device="cuda", dtype=torch.float32)
        pick = torch.multinomial(pop, B, replacement=True, generator=gen)
        shift = torch.zeros(B, d, device="cuda")
        for w in ({"Wr_att", "Wr_mlp"} if case["heads"] else {"Wr_mlp"}):
            col = routers[w].float()[:, pick].t()
            shift += case["skew"] * col / (col * col).sum(1, keepdim=True)
    state = {"case": case, "x": tokens(shift)}
    kind = case["kind"]
    if kind in ("block_fwd", "block_train"):
        std = case["w_std"]
        weights = dict(routers, Wq=normal(n, d, d_g, std=std), Wk=normal(n, d, d_g, std=std), Wv=normal(n, d, d_g, std=std),
                       Wo=normal(n, d_g, d, std=std), W1=normal(n, d, d_e, std=std), W2=normal(n, d_e, d, std=std))
        state["block"] = UoEBlock(_problem(case, "att"), _problem(case, "mlp"), weights, backward=kind == "block_train")
    elif kind == "mlp_train":
        std = case["w_std"]
        weights = {"Wr_mlp": routers["Wr_mlp"], "W1": normal(n, d, d_e, std=std), "W2": normal(n, d_e, d, std=std)}
        state["block"] = UoEBlock(None, _problem(case, "mlp"), weights, backward=True)
    elif kind == "mlp_f32":
        prob = _problem(case, "mlp")
        state.update(prob=prob, W_r=routers["Wr_mlp"], W1=normal(n, d, d_e, std=case["w_std"]), W2=normal(n, d_e, d, std=case["w_std"]),
                     b1=normal(n, d_e, std=0.1), b2=normal(n, d, std=0.1), routing=uoe.alloc_routing(prob),
                     y=torch.empty_like(state["x"]), ws_route=uoe.alloc_workspace(prob, uoe.UOE_OP_ROUTE),
                     ws=uoe.alloc_workspace(prob, uoe.UOE_OP_MLP_FWD))
    else:
        prob = _problem(case, "mlp")
        state.update(prob=prob, W_r=routers["Wr_mlp"], routing=uoe.alloc_routing(prob), dloss=torch.ones(B, device="cuda"),
                     ws_route=uoe.alloc_workspace(prob, uoe.UOE_OP_ROUTE), ws=uoe.alloc_workspace(prob, uoe.UOE_OP_BALANCE_BWD))
    if kind in ("block_train", "mlp_train"):
        state["dy"] = tokens()
    return state


def run(state):
    kind, x = state["case"]["kind"], state["x"]
    if kind == "block_fwd":
        return state["block"].forward(x)
    if kind == "block_train":
        block = state["block"]
        y = block.forward(x)
        du, dW1, dW2, dWr_mlp = block.mlp_backward(block.u, state["dy"])
        dx, dWq, dWk, dWv, dWo, dWr_att = block.smha_backward(x, du)
        return {"y": y, "dx": dx, "dW1": dW1, "dW2": dW2, "dWr_mlp": dWr_mlp, "dWq": dWq, "dWk": dWk, "dWv": dWv, "dWo": dWo,
                "dWr_att": dWr_att}
    if kind == "mlp_train":
        block = state["block"]
        y = block.forward(x)
        dx, dW1, dW2, dWr = block.mlp_backward(x, state["dy"])
        return {"y": y, "dx": dx, "dW1": dW1, "dW2": dW2, "dWr": dWr}
    if kind == "mlp_f32":
        r = uoe.uoe_route(state["prob"], x, state["W_r"], out=state["routing"], ws=state["ws_route"], check=False)
        return uoe.uoe_mlp_forward(state["prob"], x, state["W1"], state["W2"], r, b1=state["b1"], b2=state["b2"], y=state["y"],
                                   ws=state["ws"], check=False)
    prob, W_r = state["prob"], state["W_r"]
    r = uoe.uoe_route(prob, x, W_r, out=state["routing"], ws=state["ws_route"], check=False)
    loss, count, c_dyn = uoe.uoe_route_balance(prob, r.p_patch, alpha=0.01)
    dx, dW_r = uoe.uoe_route_balance_backward(prob, x, W_r, r.p_patch, 0.01, state["dloss"], ws=state["ws"])
    return {"expert_idx": r.expert_idx, "patch_idx": r.patch_idx, "gate": r.gate, "p_samp": r.p_samp, "p_patch": r.p_patch,
            "expert_offsets": r.expert_offsets, "loss": loss, "count": count, "c_dyn": c_dyn, "dx": dx, "dW_r": dW_r}


# ---------------------------------------------------------------------------------------------------------------
# what a pass cannot do without, and how far two correct passes may be apart
# ---------------------------------------------------------------------------------------------------------------

def work(case):
    B, d, n, k, d_e, d_g = case["B"], case["d"], case["n"], case["k"], case["d_e"], case["heads"] * HEAD_DIM
    esize = 4 if case["kind"] == "mlp_f32" else 2
    l_a = min(case["c"] * case["l_p"], case["L_valid"])              # tokens an expert takes of a sample
    rows = B * k * l_a
    tok = B * case["m"] * case["l_p"] * d * esize                    # one activation tensor
    route = 2.0 * B * case["L_valid"] * d                            # column sums; the dot products are negligible
    mlp = 4.0 * rows * d * d_e
    att = 2.0 * rows * d * 4 * d_g + 4.0 * rows * l_a * d_g * (0.5 if case["causal"] else 1.0)
    w_mlp, w_att = 2 * n * d * d_e, 4 * n * d * d_g
    kind = case["kind"]
    if kind == "block_fwd":
        return {"bytes": 2 * tok + (w_mlp + w_att) * esize, "flops": mlp + att + 2 * route}
    if kind == "block_train":      # x, dy read, y, dx written; weights read, their float32 gradients written
        return {"bytes": 4 * tok + (w_mlp + w_att) * (esize + 4), "flops": 3 * (mlp + att) + 4 * route}
    if kind == "mlp_train":
        return {"bytes": 4 * tok + w_mlp * (esize + 4), "flops": 3 * mlp + 2 * route}
    if kind == "mlp_f32":
        return {"bytes": 2 * tok + w_mlp * esize, "flops": mlp + route}
    return {"bytes": 2 * tok + 2 * d * n * esize, "flops": 2 * route}


def tolerance(case):
    # four times the distance from the same pass in 64 bits: forward outputs 1.2e-3 to 1.5e-3 (bfloat16 storage of y),
    # gradients 1.7e-3 to 4.2e-3 (bfloat16 operands), float32 below 1e-7 plus the room that wider drawn layers need
    kind = case["kind"]
    if kind == "mlp_f32":
        return {"rel": 1e-6}
    if kind == "router_train":      # dx is stored in bfloat16; indices may differ where two gate values tie to the last bits
        return {"rel": 7e-3, "differ": 2e-3}
    return {"rel": 6e-3 if kind == "block_fwd" else 1.7e-2}
