"""The work a user of this library has it do: the Mixture-of-Experts layer forward pass (bf16, MX FP8 and FP8
block-scaled weights; softmax and grouped sigmoid routing; all experts or a resident subset) and one decode step of
paged grouped-query attention, from single-token calls to prefill batches.

A case is a dict of plain values with a ``"kind"``:

  "layer"   T tokens, H hidden, I intermediate, E experts, top_k; ``weights`` = "bf16" | "mxfp8" | "fp8w";
            ``router`` = "softmax" | "grouped"; ``local`` resident experts from ``local_offset`` on (= E, 0 for all);
            ``skew``: Zipf-biased router logits, so that a few experts take most of the tokens
  "decode"  B sequences of len_lo..len_hi cached tokens (drawn uniformly), Hq query heads over Hkv key-value heads,
            pages of page_size tokens scattered over the cache; head dimension 128
"""
from __future__ import annotations

import math

import torch

import paper_2602_19128_b200 as moe
from paper_2602_19128_b200.inputs import make_gqa_inputs, make_inputs, zipf_bias

DEVICE = "cuda:0"


def _layer(T, H, I, E, top_k, weights="bf16", router="softmax", local=None, local_offset=0, skew=False):
    return dict(kind="layer", T=T, H=H, I=I, E=E, top_k=top_k, weights=weights, router=router,
                local=E if local is None else local, local_offset=local_offset, skew=skew)


def _decode(B, len_lo, len_hi, Hq=32, Hkv=4, page_size=16):
    return dict(kind="decode", B=B, Hq=Hq, Hkv=Hkv, page_size=page_size, len_lo=len_lo, len_hi=len_hi)


def listed():
    return [
        # The smallest layer of the benchmark: latency of the launch sequence.
        dict(name="layer_tiny", **_layer(16, 256, 512, 8, 2)),
        # Interactive generation, one sequence: a single token through a Mixtral-shaped layer.
        dict(name="layer_mixtral_t1", **_layer(1, 4096, 14336, 8, 2)),
        # A few hundred concurrent sequences (or a short prompt) through the same layer.
        dict(name="layer_mixtral_t512", **_layer(512, 4096, 14336, 8, 2)),
        # One decode step of 128 sequences, DeepSeek-V3-shaped experts all on one GPU: nearly every expert is
        # touched by a handful of tokens.
        dict(name="layer_dsv3_decode", **_layer(128, 7168, 2048, 256, 8)),
        # A prefill batch of the same model: the largest call.
        dict(name="layer_dsv3_prefill", **_layer(8192, 7168, 2048, 256, 8)),
        # Hot experts: most tokens go to a few of 128 experts, many experts get none.
        dict(name="layer_skewed", **_layer(4096, 4096, 1536, 128, 8, skew=True)),
        # Expert-parallel deployment in MX FP8: 32 of 256 experts resident, grouped routing; prefill ...
        dict(name="layer_local32_mxfp8_prefill",
             **_layer(8192, 7168, 2048, 256, 8, weights="mxfp8", router="grouped", local=32, local_offset=64)),
        # ... and decode.
        dict(name="layer_local32_mxfp8_decode",
             **_layer(128, 7168, 2048, 256, 8, weights="mxfp8", router="grouped", local=32, local_offset=64)),
        # FP8 weights with block scales under bf16 activations, an odd number of tokens.
        dict(name="layer_mixtral_fp8w_t333", **_layer(333, 4096, 14336, 8, 2, weights="fp8w")),
        # Attention of one decode step: a mixed serving batch, one long sequence, many short sequences.
        dict(name="decode_b64", **_decode(64, 1024, 8192)),
        dict(name="decode_b1_long", **_decode(1, 65536, 65536)),
        dict(name="decode_b256_short", **_decode(256, 256, 2048)),
    ]


# ---- drawn cases ---------------------------------------------------------------------------------------------
_LAYER_SHAPES = [(256, 512, 8, 2), (4096, 14336, 8, 2), (7168, 2048, 256, 8), (4096, 1536, 128, 8)]
_MAX_WEIGHTS = 256 * 3 * 7168 * 2048          # weights of the largest listed layer
_MAX_MACS = 8192 * 8 * 3 * 7168 * 2048        # and its multiply-adds


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_layer(rng):
    weights = rng.choice(["bf16", "bf16", "mxfp8", "mxfp8", "fp8w"])
    while True:
        if rng.random() < 0.5:
            H, I, E, k = rng.choice(_LAYER_SHAPES)
        else:
            H = 256 * _log_int(rng, 1, 28)
            I = (64 if weights == "bf16" else 128) * _log_int(rng, 4, 64)
            E = rng.choice([8, 16, 20, 32, 60, 64, 128, 160, 256])
            k = rng.choice([1, 2, 4, 6, 8])
        router = rng.choice(["softmax", "grouped"]) if E in (64, 128, 256) and weights != "fp8w" else "softmax"
        parts = rng.choice([1, 1, 2, 8]) if weights != "fp8w" and E % 8 == 0 else 1
        local = E // parts
        T = _log_int(rng, 1, 8192)
        if T > 16 and rng.random() < 0.5:
            T |= 1
        if local * 3 * H * I <= _MAX_WEIGHTS and T * k * 3 * H * I <= parts * _MAX_MACS:
            return _layer(T, H, I, E, k, weights, router, local, local * rng.randrange(parts),
                          skew=router == "softmax" and parts == 1 and rng.random() < 0.25)


def _draw_decode(rng):
    while True:
        B = _log_int(rng, 1, 256)
        hi = _log_int(rng, 128, 65536)
        Hq, Hkv = rng.choice([(32, 4), (32, 4), (32, 8), (16, 2), (64, 8), (8, 8), (24, 8)])
        if B * hi * Hkv <= 64 * 16384 * 4:
            return _decode(B, max(1, hi // rng.choice([1, 2, 8])), hi, Hq, Hkv, rng.choice([1, 8, 16, 16, 32, 64]))


def draw(rng):
    return _draw_decode(rng) if rng.random() < 0.3 else _draw_layer(rng)


# ---- what a program holds before the call --------------------------------------------------------------------
def _quantize_blocks(w):
    """E4M3 codes and one fp32 scale (amax / 448) per 128 x 128 block of each expert's matrix."""
    E, R, C = w.shape
    codes = torch.empty((E, R, C), dtype=torch.uint8, device=w.device)
    scales = torch.empty((E, R // 128, C // 128), dtype=torch.float32, device=w.device)
    for e in range(E):
        blocks = w[e].float().view(R // 128, 128, C // 128, 128)
        scales[e] = (blocks.abs().amax(dim=(1, 3)) / 448.0).clamp_min(1e-12)
        codes[e] = (blocks / scales[e][:, None, :, None]).to(torch.float8_e4m3fn).view(torch.uint8).view(R, C)
    return codes, scales


def _quantize_mx(w, gate_up):
    """MX FP8 codes and packed scale bytes, as a program prepares them once per model."""
    E, R, K = w.shape
    codes, scales = moe.moe_mxfp8_quantize_rows(w.view(E * R, K))
    return codes.view(E, R, K), moe.moe_mxfp8_pack_scales(scales.view(E, R, K // 32), gate_up)


def _prepare_layer(case, seed):
    inp = make_inputs(case, seed=seed, device=DEVICE)
    T, H, I, E, k = (case[n] for n in ("T", "H", "I", "E", "top_k"))
    st = dict(case=case, x=inp["x"], logits=inp["router_logits"], out=torch.empty_like(inp["x"]), router=None)
    if case["router"] == "grouped":
        gen = torch.Generator(device=DEVICE)
        gen.manual_seed(seed + 1)
        # a small correction bias, as load balancing leaves it
        st["bias"] = 0.02 * torch.randn(E, generator=gen, device=DEVICE, dtype=torch.float32)
        st["router"] = moe.grouped_router(8, 4, st["bias"], 2.5)
    if case["weights"] == "mxfp8":
        st["weights"] = _quantize_mx(inp.pop("w13"), True) + _quantize_mx(inp.pop("w2"), False)
        nbytes = moe.moe_mxfp8_workspace_bytes(T, H, I, E, k)
    else:
        if case["weights"] == "fp8w":
            st["weights"] = _quantize_blocks(inp.pop("w13")) + _quantize_blocks(inp.pop("w2"))
        else:
            st["weights"] = (inp["w13"], inp["w2"])
        nbytes = moe.moe_workspace_bytes(T, H, I, E, k)
    st["workspace"] = moe.alloc_workspace(nbytes, DEVICE)
    return st


def _prepare_decode(case, seed):
    inp = make_gqa_inputs(dict(case, D=128), seed=seed, device=DEVICE)
    max_len = max(inp["kv_len"])
    nbytes = moe.gqa_decode_workspace_bytes(case["B"], case["Hq"], case["Hkv"], 128, max_len)
    return dict(case=case, inp=inp, max_len=max_len, out=torch.empty_like(inp["q"]),
                lse=torch.empty((case["B"], case["Hq"]), dtype=torch.float32, device=DEVICE),
                workspace=moe.alloc_workspace(nbytes, DEVICE))


def prepare(case, seed):
    return _prepare_layer(case, seed) if case["kind"] == "layer" else _prepare_decode(case, seed)


# ---- one pass ------------------------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    if case["kind"] == "decode":
        inp = state["inp"]
        moe.gqa_paged_decode(inp["q"], inp["k_cache"], inp["v_cache"], inp["kv_indptr"], inp["kv_indices"],
                             inp["kv_last_page_len"], state["max_len"], inp["sm_scale"], state["out"], state["workspace"],
                             lse=state["lse"])
        return state["out"], state["lse"]
    x, logits, k, out, ws = state["x"], state["logits"], case["top_k"], state["out"], state["workspace"]
    router, lo = state["router"], case["local_offset"]
    if case["weights"] == "mxfp8":
        moe.moe_forward_mxfp8(x, logits, *state["weights"], k, out, ws, local_expert_offset=lo, router=router)
    elif case["weights"] == "fp8w":
        moe.moe_forward_fp8w(x, logits, *state["weights"], k, out, ws)
    elif router is not None:
        moe.moe_forward_grouped(x, logits, *state["weights"], k, router, out, ws, local_expert_offset=lo)
    elif case["local"] < case["E"]:
        moe.moe_forward_local(x, logits, *state["weights"], k, lo, out, ws)
    else:
        moe.moe_forward(x, logits, *state["weights"], k, out, ws)
    return out


# ---- what one pass cannot do without -------------------------------------------------------------------------
def _active_experts(case):
    """Expected number of resident experts that at least one token selects."""
    T, E, k = case["T"], case["E"], case["top_k"]
    if not case["skew"]:
        return case["local"] * (1.0 - (1.0 - k / E) ** T)
    gen = torch.Generator()
    gen.manual_seed(0)
    logits = torch.randn((T, E), generator=gen) + zipf_bias(E)
    return float(torch.unique(logits.topk(k, dim=1).indices).numel())


def work(case):
    if case["kind"] == "decode":
        tokens = case["B"] * (case["len_lo"] + case["len_hi"]) / 2
        q = case["B"] * case["Hq"] * 128
        pages = tokens / case["page_size"]
        return {"bytes": int(tokens * case["Hkv"] * 128 * 2 * 2 + 2 * q * 2 + case["B"] * (case["Hq"] + 2) * 4 + pages * 4),
                "flops": int(4 * tokens * case["Hq"] * 128)}
    T, H, I, E, k = (case[n] for n in ("T", "H", "I", "E", "top_k"))
    per_weight = {"bf16": 2.0, "mxfp8": 1.0 + 1.0 / 32, "fp8w": 1.0 + 4.0 / 128 ** 2}[case["weights"]]
    return {"bytes": int(_active_experts(case) * 3 * H * I * per_weight + T * (2 * H * 2 + E * 4)),
            "flops": int(6 * T * k * case["local"] / E * H * I)}


def tolerance(case):
    """About four times the largest error seen against a reference with its sums in another order (fp32 library
    products with the layer's own roundings, for bf16 and FP8 weights 1.4e-3, for MX FP8 4e-4; for the attention step
    float64 without intermediate roundings, 2.2e-3)."""
    if case["kind"] == "decode":
        return {"rel": 9e-3}
    return {"rel": 1.6e-3 if case["weights"] == "mxfp8" else 5.5e-3}
