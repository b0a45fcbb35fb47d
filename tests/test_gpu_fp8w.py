"""GPU parity of moe_forward_fp8w (FP8 E4M3 block-scaled expert weights) against the oracle."""
import numpy as np
import pytest
import torch

import paper_2602_19128_b200 as moe
from oracle import moe_oracle
from paper_2602_19128_b200.inputs import bf16_bits
from tests.weight_quantizers import make_fp8w_inputs
from tests.gpu_common import (Guarded, assert_close_out, assert_routing_exact, assert_same_bits_again, bf16_to_f64, check_guards,
                              guarded_out, layer_regions, widen_hidden)

pytestmark = pytest.mark.gpu


def call_fp8w(inp, out, ws):
    moe.moe_forward_fp8w(inp["x"], inp["router_logits"], inp["w13_q"], inp["w13_scale"], inp["w2_q"], inp["w2_scale"],
                         inp["top_k"], out, ws)


def assert_fp8w_same_bits_again(inp, out):
    (T, H), (E, I2, _), k = inp["x"].shape, inp["w13_q"].shape, inp["top_k"]
    ws = moe.alloc_workspace(moe.moe_workspace_bytes(T, H, I2 // 2, E, k), "cuda")
    assert_same_bits_again(lambda o, w: call_fp8w(inp, o, w), out, ws, moe.moe_workspace_layout(T, H, I2 // 2, E, k).topk_ids)


def run_fp8w(inp):
    T, H = inp["x"].shape
    E, I2, _ = inp["w13_q"].shape
    I, k = I2 // 2, inp["top_k"]
    wg = Guarded(moe.moe_workspace_bytes(T, H, I, E, k), "cuda")
    ws = wg.inner
    og, out = guarded_out(T, H, "cuda")
    call_fp8w(inp, out, ws)
    assert moe.moe_last_status(ws) == moe.MOE_OK
    check_guards(wg, og, moe.moe_workspace_layout(T, H, I, E, k), layer_regions(T, H, I, E, k), "moe_forward_fp8w")
    return out, moe.workspace_views(ws, T, H, I, E, k)


def oracle_out(inp):
    o = moe_oracle.get("f32")
    return o.forward_fp8w(bf16_bits(inp["x"]), inp["router_logits"].cpu().numpy(), inp["w13_q"].cpu().numpy(),
                          inp["w13_scale"].cpu().numpy(), inp["w2_q"].cpu().numpy(), inp["w2_scale"].cpu().numpy(),
                          inp["top_k"])


# T, H, I, E, k, skew: every token-tile bound (32..256), several K blocks, gate/up rows in different scale blocks
CASES = [
    (16, 256, 512, 8, 2, False),
    (1, 128, 128, 4, 1, False),
    (128, 384, 128, 256, 8, False),   # decode-like, N = 16
    (200, 256, 384, 8, 2, False),     # ~50 rows per expert
    (300, 128, 128, 64, 4, True),     # skewed, empty experts
    (700, 256, 256, 4, 2, False),     # two token tiles per expert, N up to 256
    (96, 128, 256, 8, 8, False),
]


@pytest.mark.parametrize("T,H,I,E,k,skew", CASES)
def test_fp8w_forward_matches_oracle(T, H, I, E, k, skew):
    inp = make_fp8w_inputs(dict(T=T, H=H, I=I, E=E, top_k=k, skew=skew), seed=0, device="cuda")
    out, views = run_fp8w(inp)
    o = moe_oracle.get("f32")
    ids, w = o.route(inp["router_logits"].cpu().numpy(), k)
    off, s2f, f2s = o.permute(ids, E)
    assert_routing_exact(views, ids, w, off, s2f, f2s)
    assert_close_out(bf16_to_f64(out), oracle_out(inp), "fp8w out")


@pytest.mark.parametrize("T,H,I,E,k", [(8, 2048, 1408, 2, 2),    # tiles of up to 32 rows, 16 and 11 slots of K
                                       (31, 1920, 1152, 2, 2),   # 64: 15 and 9 slots
                                       (75, 1408, 2048, 2, 2),   # 128
                                       (190, 1664, 1280, 2, 2),  # 192, one tile per expert
                                       (193, 896, 1152, 2, 2)])  # 192, two ragged tiles per expert
def test_fp8w_long_rows_wrap_the_rings(T, H, I, E, k):
    """K longer than the weight ring and the operand buffers, slot counts that are no multiple of either: every buffer
    is reused across tiles in another phase."""
    inp = make_fp8w_inputs(dict(T=T, H=H, I=I, E=E, top_k=k, skew=False), seed=3, device="cuda")
    out, _ = run_fp8w(inp)
    assert_close_out(bf16_to_f64(out), oracle_out(inp), "fp8w out")


@pytest.mark.parametrize("T,H,I,E,k,skew", [(70, 1280, 1024, 2, 2, False),    # tiles of up to 128 rows, 10 and 8 slots of K
                                            (75, 1024, 1408, 2, 2, False),    # 8 and 11
                                            (190, 1280, 1152, 2, 2, False),   # 192, one tile per expert
                                            (193, 1024, 1152, 2, 2, False),   # 192, two ragged tiles per expert
                                            (300, 1024, 1024, 16, 4, True)])  # skewed: from many tiles per expert to none
def test_fp8w_cta_pairs_for_both_gemms(T, H, I, E, k, skew):
    """K loops of eight slots and more and whole pair tiles of features: both GEMMs run on CTA pairs."""
    inp = make_fp8w_inputs(dict(T=T, H=H, I=I, E=E, top_k=k, skew=skew), seed=5, device="cuda")
    out, _ = run_fp8w(inp)
    assert_close_out(bf16_to_f64(out), oracle_out(inp), "fp8w out")


@pytest.mark.parametrize("T,H,I,E,k", [(1, 512, 2048, 4, 2), (3, 256, 2176, 2, 2), (30, 384, 2304, 4, 2)])
def test_fp8w_few_down_tiles_with_two_ctas_each(T, H, I, E, k):
    """Two CTAs per tile of the down GEMM, half of its rows each (2176: 17 slots); the same bits as with one CTA per tile,
    which the layer has with its hidden dimension padded (tests/test_gpu_forward.py)."""
    inp = make_fp8w_inputs(dict(T=T, H=H, I=I, E=E, top_k=k, skew=False), seed=6, device="cuda")
    out, _ = run_fp8w(inp)
    assert_close_out(bf16_to_f64(out), oracle_out(inp), "fp8w out")
    to = 5120
    w = widen_hidden(inp["x"], w13=inp["w13_q"], w2=inp["w2_q"], to=to)
    blocks = torch.arange(to // 128, device="cuda") % (H // 128)
    wide = dict(inp, x=w["x"], w13_q=w["w13"], w2_q=w["w2"], w2_scale=inp["w2_scale"][:, blocks].contiguous(),
                w13_scale=torch.nn.functional.pad(inp["w13_scale"], (0, (to - H) // 128), value=1.0))
    out_wide, _ = run_fp8w(wide)
    assert torch.equal(out.view(torch.int16), out_wide[:, :H].view(torch.int16))


@pytest.mark.parametrize("T,H,I,E,k", [(40, 256, 1152, 16, 2),    # 18 slabs of 16 experts and more: two launches in sequence
                                       (300, 896, 4096, 18, 2),   # 7 slots, more than seven rounds: the same
                                       (24, 256, 256, 8, 2),      # one round: the down GEMM starts through the hand-over
                                       (40, 2048, 256, 16, 2)])   # 16 slots: the same
def test_fp8w_with_and_without_the_hand_over(T, H, I, E, k):
    """Both ways from the gate/up GEMM to the down GEMM, and a second call in the same workspace after each."""
    inp = make_fp8w_inputs(dict(T=T, H=H, I=I, E=E, top_k=k, skew=False), seed=4, device="cuda")
    out, _ = run_fp8w(inp)
    assert_close_out(bf16_to_f64(out), oracle_out(inp), "fp8w out")
    ws = moe.alloc_workspace(moe.moe_workspace_bytes(T, H, I, E, k), "cuda")
    for _ in range(2):
        again = torch.empty_like(out)
        moe.moe_forward_fp8w(inp["x"], inp["router_logits"], inp["w13_q"], inp["w13_scale"], inp["w2_q"], inp["w2_scale"], k,
                             again, ws)
        assert torch.equal(out.view(torch.int16), again.view(torch.int16))


@pytest.mark.parametrize("T,H,I,E,k,skew", [(64, 256, 2048, 64, 4, False),   # 32-row tiles, 14 per CTA, two slots each
                                            (150, 256, 2048, 32, 8, True),   # 64 rows, ragged
                                            (300, 128, 2048, 16, 4, False),  # 128 rows, one slot
                                            (900, 384, 2048, 8, 1, True)])   # 192 rows, three slots
def test_fp8w_many_short_tiles_per_cta(T, H, I, E, k, skew):
    """More tiles per CTA than the queue of decoded tiles holds, with fewer slots of K than there are operand buffers."""
    inp = make_fp8w_inputs(dict(T=T, H=H, I=I, E=E, top_k=k, skew=skew), seed=7, device="cuda")
    out, _ = run_fp8w(inp)
    assert_close_out(bf16_to_f64(out), oracle_out(inp), "fp8w out")


@pytest.mark.parametrize("T,H,I,E,k,skew", [(24, 3072, 3200, 8, 2, False),    # 32-row tiles, 24 and 25 slots of K
                                            (60, 2560, 2688, 8, 4, True)])    # 64 rows, 20 and 21 slots
def test_fp8w_tiles_on_demand(T, H, I, E, k, skew):
    """Long tiles and more than one per CTA in both GEMMs."""
    inp = make_fp8w_inputs(dict(T=T, H=H, I=I, E=E, top_k=k, skew=skew), seed=8, device="cuda")
    out, _ = run_fp8w(inp)
    assert_close_out(bf16_to_f64(out), oracle_out(inp), "fp8w out")
    assert_fp8w_same_bits_again(inp, out)


def test_fp8w_with_unit_scales_equals_the_bf16_layer_bit_for_bit():
    """All E4M3 values are bf16 values, and a scale of 1 is exact in bf16: both paths see the same operands."""
    g = torch.Generator().manual_seed(0)
    T, H, I, E, k = 64, 256, 128, 4, 2
    table = torch.arange(256, dtype=torch.uint8).view(torch.float8_e4m3fn).float()
    finite = torch.nonzero(~torch.isnan(table) & (table.abs() <= 1.0)).flatten()
    c13 = finite[torch.randint(len(finite), (E, 2 * I, H), generator=g)].to(torch.uint8).cuda()
    c2 = finite[torch.randint(len(finite), (E, H, I), generator=g)].to(torch.uint8).cuda()
    inp = dict(x=(torch.randn(T, H, generator=g) * 0.05).to(torch.bfloat16).cuda(),
               router_logits=torch.randn(T, E, generator=g).cuda(), top_k=k, w13_q=c13, w2_q=c2,
               w13_scale=torch.ones(E, 2 * I // 128, H // 128, device="cuda"),
               w2_scale=torch.ones(E, H // 128, I // 128, device="cuda"))
    out, _ = run_fp8w(inp)
    w13 = table.cuda()[c13.long()].to(torch.bfloat16)
    w2 = table.cuda()[c2.long()].to(torch.bfloat16)
    ref = torch.empty_like(out)
    ws = moe.alloc_workspace(moe.moe_workspace_bytes(T, H, I, E, k), "cuda")
    moe.moe_forward(inp["x"], inp["router_logits"], w13, w2, k, ref, ws, flags=moe.MOE_FLAG_SINGLE_CTA_GEMM)
    torch.cuda.synchronize()
    assert torch.equal(out.view(torch.int16), ref.view(torch.int16))


def test_fp8w_pair_tiles_on_demand():
    """80 slots of K and 80 tiles of the down GEMM on 74 pairs, against the bf16 layer on the same values (unit scales: the same
    bits), and again and again in one workspace."""
    g = torch.Generator(device="cuda").manual_seed(1)
    T, H, I, E, k = 300, 2560, 10240, 8, 2
    table = torch.arange(256, dtype=torch.uint8).view(torch.float8_e4m3fn).float()
    finite = torch.nonzero(~torch.isnan(table) & (table.abs() <= 0.125)).flatten().to(torch.uint8).cuda()
    codes = lambda *shape: finite[torch.randint(len(finite), shape, generator=g, device="cuda")]
    c13, c2 = codes(E, 2 * I, H), codes(E, H, I)
    inp = dict(x=(torch.randn(T, H, generator=g, device="cuda") * 0.1).to(torch.bfloat16),
               router_logits=torch.randn(T, E, generator=g, device="cuda"), top_k=k, w13_q=c13, w2_q=c2,
               w13_scale=torch.ones(E, 2 * I // 128, H // 128, device="cuda"), w2_scale=torch.ones(E, H // 128, I // 128, device="cuda"))
    out, ws = run_fp8w(inp)
    values = table.to(torch.bfloat16).cuda()
    ref = torch.empty_like(out)
    moe.moe_forward(inp["x"], inp["router_logits"], torch.stack([values[c.int()] for c in c13]), torch.stack([values[c.int()] for c in c2]), k, ref,
                    moe.alloc_workspace(moe.moe_workspace_bytes(T, H, I, E, k), "cuda"), flags=moe.MOE_FLAG_SINGLE_CTA_GEMM)
    torch.cuda.synchronize()
    assert torch.isfinite(ref.float()).all() and torch.equal(out.view(torch.int16), ref.view(torch.int16))
    assert_fp8w_same_bits_again(inp, out)


def test_fp8w_rejects_shapes_outside_its_envelope():
    inp = make_fp8w_inputs(dict(T=8, H=128, I=128, E=2, top_k=1, skew=False), seed=1, device="cuda")
    out = torch.zeros((8, 128), dtype=torch.bfloat16, device="cuda")
    ws = moe.alloc_workspace(1 << 20, "cuda")
    bad_q = torch.zeros((2, 2 * 192, 128), dtype=torch.uint8, device="cuda")     # I = 192 is not a multiple of 128
    bad_s = torch.ones((2, 3, 1), device="cuda")
    bad_q2 = torch.zeros((2, 128, 192), dtype=torch.uint8, device="cuda")
    assert moe.moe_forward_fp8w(inp["x"], inp["router_logits"], bad_q, bad_s, bad_q2, bad_s, 1, out, ws, check=False) == -3
