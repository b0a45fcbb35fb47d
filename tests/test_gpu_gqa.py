"""GPU parity of the second workload, paged grouped-query decode attention (include/gqa_decode.h), against the
double-precision CPU oracle, element by element, through the C ABI.

Tolerance: |gpu - oracle| <= 1e-2 * (1 + |oracle|) for every output element and 2e-3 for lse.  The kernel rounds the
probabilities to bf16 for the P V product (relative 2^-9 each, averaging out over the tokens) and the result to bf16
(relative 2^-9); scores and sums are fp32.  Outputs are O(1), so the bound is several times the expected error."""
import numpy as np
import pytest
import torch

import paper_2602_19128_b200 as moe
from oracle import gqa_oracle
from paper_2602_19128_b200.inputs import GQA_CONFIGS, bf16_bits, make_gqa_inputs
from tests.gpu_common import Guarded

pytestmark = pytest.mark.gpu

OUT_TOL, LSE_TOL = 1e-2, 2e-3


def run_gpu(inp, max_kv_len=None, want_lse=True):
    B, Hq, Hkv, D = inp["B"], inp["Hq"], inp["Hkv"], inp["D"]
    max_kv_len = max(inp["kv_len"] + [0]) if max_kv_len is None else max_kv_len
    wg = Guarded(moe.gqa_decode_workspace_bytes(B, Hq, Hkv, D, max_kv_len), "cuda")
    og = Guarded(B * Hq * D * 2, "cuda")
    out = og.inner[:B * Hq * D * 2].view(torch.bfloat16).view(B, Hq, D)
    lg = Guarded(B * Hq * 4, "cuda")
    lse = lg.inner[:B * Hq * 4].view(torch.float32).view(B, Hq) if want_lse else None
    moe.gqa_paged_decode(inp["q"], inp["k_cache"], inp["v_cache"], inp["kv_indptr"], inp["kv_indices"],
                         inp["kv_last_page_len"], max_kv_len, inp["sm_scale"], out, wg.inner, lse=lse)
    torch.cuda.synchronize()
    for g, name in ((wg, "workspace"), (og, "out"), (lg, "lse")):
        g.assert_bands_intact(f"gqa_paged_decode {name}")
    return out, lse


def oracle(inp):
    return gqa_oracle.get("f64").paged_decode(bf16_bits(inp["q"]), bf16_bits(inp["k_cache"]), bf16_bits(inp["v_cache"]),
                                              inp["kv_indptr"].cpu().numpy(), inp["kv_indices"].cpu().numpy(),
                                              inp["kv_last_page_len"].cpu().numpy(), inp["sm_scale"])


def check(inp, max_kv_len=None):
    out, lse = run_gpu(inp, max_kv_len)
    ref, ref_lse = oracle(inp)
    got = out.float().cpu().numpy().astype(np.float64)
    assert np.isfinite(got).all()
    err, bound = np.abs(got - ref), OUT_TOL * (1 + np.abs(ref))
    worst = np.unravel_index(np.argmax(err - bound), err.shape)
    assert (err <= bound).all(), f"out worst at {worst}: gpu={got[worst]} ref={ref[worst]}"
    got_lse = lse.cpu().numpy().astype(np.float64)
    empty = np.isneginf(ref_lse)
    assert np.array_equal(np.isneginf(got_lse), empty)
    assert np.abs(got_lse[~empty] - ref_lse[~empty]).max(initial=0) <= LSE_TOL
    return out


# B, Hq, Hkv, page size, lengths: chunk and split edges, ragged last pages, empty items, every group size
CASES = [
    (3, 8, 2, 4, [5, 60, 64]),
    (4, 32, 4, 16, [1, 63, 65, 129]),                 # the paper's head geometry; 64-token chunk edges
    (2, 4, 4, 1, [17, 300]),                          # one token per page; groups of one head
    (3, 16, 1, 8, [0, 5, 700]),                       # an item with nothing cached; a group of 16 heads
    (2, 6, 2, 16, [1024, 2047]),                      # groups of three; several splits per sequence
    (1, 32, 4, 16, [20000]),                          # one long sequence: many splits merged by the last block
    (5, 32, 4, 32, [16, 32, 33, 4096, 257]),          # mixed lengths: some sequences use one split, some many
    (40, 8, 4, 16, [100 + 37 * i for i in range(40)]),  # enough items that every sequence is a single split
    (2, 2, 1, 64, [64, 6000]),                        # groups of two, large pages
    (3, 32, 4, 8, [7, 1000, 5000]),                   # the smallest page the tiled gather takes: 32 boxes per chunk
    (2, 32, 4, 128, [100, 7000]),                     # pages larger than a chunk: boxes start inside a page
    (2, 8, 1, 256, [255, 9000]),
    (3, 32, 4, 12, [11, 1000, 5000]),                 # page sizes that are no power of two: the row gather
    (2, 16, 2, 3, [2, 4100]),
    (2, 32, 4, 24, [24, 6001]),
    (2, 32, 4, 2, [3000, 1]),
]


@pytest.mark.parametrize("B,Hq,Hkv,P,lengths", CASES, ids=[f"B{c[0]}h{c[1]}kv{c[2]}p{c[3]}" for c in CASES])
def test_decode_matches_oracle(B, Hq, Hkv, P, lengths):
    inp = make_gqa_inputs(dict(B=B, Hq=Hq, Hkv=Hkv, D=128, page_size=P, lengths=lengths), seed=B + Hq, device="cuda")
    check(inp)


@pytest.mark.parametrize("B,Hq,Hkv,P,long,short", [
    (24, 64, 8, 16, [8000, 0, 4100, 64], 65),     # one sequence in dozens of parts, empty items, pieces of whole sequences
    (24, 8, 8, 8, [0, 0, 8191], 1),               # groups of one head, the line starts behind empty items
    (140, 32, 2, 64, [6000, 2049, 0], 63),        # groups of 16 heads, more items than the 128 ranges they are summed in
    (300, 2, 1, 32, [9000, 128], 0),              # nearly everything empty: too many fixed shares for equal pieces
    (250, 2, 1, 32, [9000, 128], 0),              # nearly everything empty: fewer pieces than blocks
])
def test_equal_pieces_of_a_ragged_batch_match_oracle(B, Hq, Hkv, P, long, short):
    """Lengths ragged enough for the balanced form: sequences cut by the blocks' pieces at any chunk."""
    lengths = [short] * B
    for i, n in enumerate(long):
        lengths[(i * 7 + (0 if i % 2 else B - 1)) % B] = n
    inp = make_gqa_inputs(dict(B=B, Hq=Hq, Hkv=Hkv, D=128, page_size=P, lengths=lengths), seed=B, device="cuda")
    full = check(inp)
    assert ran_equal_pieces(inp) == (B != 300)
    check(inp, max_kv_len=64)   # a hint far below the lengths: one fixed share per sequence, whatever its length
    assert not ran_equal_pieces(inp, max_kv_len=64)
    again, _ = run_gpu(inp)
    assert torch.equal(full.view(torch.int16), again.view(torch.int16))   # the merge order does not depend on arrival


def ran_equal_pieces(inp, max_kv_len=None, workspace_bytes=None):
    """Whether the call cut the batch into equal pieces (the workspace's fourth word); its result is checked."""
    B, Hq, Hkv, D = inp["B"], inp["Hq"], inp["Hkv"], inp["D"]
    max_kv_len = max(inp["kv_len"]) if max_kv_len is None else max_kv_len
    wg = Guarded(moe.gqa_decode_workspace_bytes(B, Hq, Hkv, D, max_kv_len) if workspace_bytes is None else workspace_bytes, "cuda")
    out = torch.empty((B, Hq, D), dtype=torch.bfloat16, device="cuda")
    moe.gqa_paged_decode(inp["q"], inp["k_cache"], inp["v_cache"], inp["kv_indptr"], inp["kv_indices"],
                         inp["kv_last_page_len"], max_kv_len, inp["sm_scale"], out, wg.inner)
    assert moe.moe_last_status(wg.inner) == 0
    wg.assert_bands_intact("gqa_paged_decode workspace")
    ref, _ = oracle(inp)
    assert (np.abs(out.float().cpu().numpy() - ref) <= OUT_TOL * (1 + np.abs(ref))).all()
    return bool(wg.inner[12:16].view(torch.int32).item())


@pytest.mark.parametrize("B,Hkv,n,max_kv_len", [(16, 4, 1000, 16000), (30, 4, 500, 2500), (24, 8, 1000, 2500)])
def test_an_item_without_tokens_does_not_change_the_form(B, Hkv, n, max_kv_len):
    """Equal lengths keep the fixed shares, however far below the hint; so do they with one empty item among them."""
    for lengths in ([n] * B, [n] * (B - 1) + [0]):
        inp = make_gqa_inputs(dict(B=B, Hq=8 * Hkv, Hkv=Hkv, D=128, page_size=16, lengths=lengths), seed=B, device="cuda")
        assert not ran_equal_pieces(inp, max_kv_len)


@pytest.mark.parametrize("Hkv,lengths,max_kv_len", [
    (1, [30000, 0, 0, 29000], 60000),                  # empty items between, half of the splits of the others empty
    (4, [0, 20000], 40000),                            # the shares start behind an empty item
    (4, [0, 0, 0, 700, 64, 0, 1, 0], 20000),           # one short share per sequence, far below the hint
    (2, [2990 + i % 7 for i in range(131)] + [0] * 9, 3000),   # more items than the 128 ranges they are summed in
    (4, [0] * 8, 20000),                               # nothing cached at all
])
def test_shares_of_a_batch_that_leaves_some_empty_match_oracle(Hkv, lengths, max_kv_len):
    """The fixed form of a batch with empty items and with splits no sequence reaches: the blocks take the shares that
    have tokens one after the other, whatever the hint, and write the results of empty items."""
    B = len(lengths)
    inp = make_gqa_inputs(dict(B=B, Hq=4 * Hkv, Hkv=Hkv, D=128, page_size=16, lengths=lengths), seed=B, device="cuda")
    if not any(lengths):
        inp["kv_indices"] = torch.zeros(1, dtype=torch.int32, device="cuda")   # (an empty tensor has no address)
    check(inp, max_kv_len)
    assert not ran_equal_pieces(inp, max_kv_len)


def test_stages_refilled_behind_a_zeroed_tail_hold_the_next_sequence():
    """Equal pieces of many short sequences with ragged ends: nearly every stage whose last value rows were zeroed is
    filled again by the same block.  A zero that lands on the next sequence's values would change a result."""
    lengths = [6100] + [64 * (i % 3 + 1) + (7 * i) % 63 + 1 for i in range(47)]
    inp = make_gqa_inputs(dict(B=48, Hq=32, Hkv=4, D=128, page_size=16, lengths=lengths), seed=1, device="cuda")
    first = check(inp)
    assert ran_equal_pieces(inp)
    for _ in range(10):
        again, _ = run_gpu(inp)
        assert torch.equal(first.view(torch.int16), again.view(torch.int16))


@pytest.mark.parametrize("B,Hkv,long,short", [(24, 8, 8000, 65), (64, 4, 8192, 1024), (250, 1, 9000, 0)])
def test_a_workspace_of_the_fixed_splits_results_is_enough(B, Hkv, long, short):
    """The documented size makes room for equal pieces; the size that holds one partial result per fixed split (as sized
    before there were pieces) is accepted, keeps the fixed form and its bounds, and a byte less than that is refused."""
    Hq = 2 * Hkv
    inp = make_gqa_inputs(dict(B=B, Hq=Hq, Hkv=Hkv, D=128, page_size=16, lengths=[short] * (B - 1) + [long]), seed=B, device="cuda")
    n_splits = -(-long // moe.gqa_decode_split_tokens(B, Hq, Hkv, 128, long))
    up = lambda v: (v + 255) // 256 * 256
    least = 512 + up(B * Hkv * 4) + up(B * Hkv * n_splits * 2 * 8) + up(B * Hkv * n_splits * 2 * 512)
    assert least < moe.gqa_decode_workspace_bytes(B, Hq, Hkv, 128, long)
    assert ran_equal_pieces(inp)
    assert not ran_equal_pieces(inp, workspace_bytes=least)
    out = torch.zeros((B, Hq, 128), dtype=torch.bfloat16, device="cuda")
    ws = moe.alloc_workspace(least, "cuda")
    assert moe.gqa_paged_decode(inp["q"], inp["k_cache"], inp["v_cache"], inp["kv_indptr"], inp["kv_indices"],
                                inp["kv_last_page_len"], long, inp["sm_scale"], out, ws[:least - 1], check=False) == -5
    torch.cuda.synchronize()
    assert (out == 0).all()


@pytest.mark.parametrize("P", [16, 12, 64, 128])
def test_slots_past_the_end_of_a_sequence_are_never_used(P):
    """The cache behind the last token of a sequence, and every page no sequence owns, holds NaN: the tiled gather
    copies whole pages into shared memory and must still keep those values out of the result."""
    lengths = [1, P + 1, 5 * P - 1, 3000 + P // 2, 64 * 7 + 5]
    inp = make_gqa_inputs(dict(B=len(lengths), Hq=32, Hkv=4, D=128, page_size=P, lengths=lengths), seed=P, device="cuda")
    owned = torch.zeros((inp["num_pages"], P), dtype=torch.bool, device="cuda")
    indptr, indices = inp["kv_indptr"].tolist(), inp["kv_indices"]
    for b, n in enumerate(lengths):
        pages = indices[indptr[b]:indptr[b + 1]].long()
        flat = torch.zeros(len(pages) * P, dtype=torch.bool, device="cuda")
        flat[:n] = True
        owned[pages] = flat.view(len(pages), P)
    for cache in (inp["k_cache"], inp["v_cache"]):
        cache[~owned] = float("nan")
    check(inp)


@pytest.mark.parametrize("P,lengths", [
    (16, [300, 5]),                        # one part per sequence
    (16, [20000, 9000]),                   # fixed splits, merged
    (12, [20000, 9000]),                   # the same from the row gather
    (16, [8000, 3000] + [70] * 22),        # equal pieces
])
def test_nan_scores_reach_out_and_lse(P, lengths):
    """A query head of NaN, and a run of NaN keys long enough to be whole parts of the sequence: out and lse are NaN
    for the heads that saw them, whether a sequence was merged from parts or not.  (lse = -inf would say that nothing
    is cached: a caller that combines attention states by lse would drop the NaN.)"""
    inp = make_gqa_inputs(dict(B=len(lengths), Hq=32, Hkv=4, D=128, page_size=P, lengths=lengths), seed=P, device="cuda")
    expect_out, expect_lse = oracle(inp)
    nan = np.zeros(expect_lse.shape, dtype=bool)
    inp["q"][0, 3] = float("nan")
    nan[0, 3] = True
    n_pages = min(lengths[0] // P, 6000 // P)           # the first tokens of item 0, as whole pages, key-value head 2
    inp["k_cache"][inp["kv_indices"][:n_pages].long(), :, 2] = float("nan")
    nan[0, 16:24] = True
    out, lse = run_gpu(inp)
    got, got_lse = out.float().cpu().numpy(), lse.cpu().numpy()
    assert np.array_equal(np.isnan(got_lse), nan), got_lse[0]
    assert np.isnan(got[nan]).all()
    assert (np.abs(got - expect_out) <= OUT_TOL * (1 + np.abs(expect_out)))[~nan].all()
    assert (np.abs(got_lse - expect_lse) <= LSE_TOL)[~nan].all()


def test_the_workspace_status_word_reports_success():
    inp = make_gqa_inputs(dict(B=2, Hq=32, Hkv=4, D=128, page_size=16, lengths=[5000, 300]), seed=3, device="cuda")
    ws = moe.alloc_workspace(moe.gqa_decode_workspace_bytes(2, 32, 4, 128, 5000), "cuda")
    ws.fill_(0x5A)
    out = torch.empty((2, 32, 128), dtype=torch.bfloat16, device="cuda")
    moe.gqa_paged_decode(inp["q"], inp["k_cache"], inp["v_cache"], inp["kv_indptr"], inp["kv_indices"],
                         inp["kv_last_page_len"], 5000, inp["sm_scale"], out, ws)
    assert moe.moe_last_status(ws) == 0


def test_an_expired_barrier_wait_is_reported_and_leaves_the_device_usable():
    """Every wait of the kernel is bounded.  The self-test waits a few milliseconds on a barrier at which nothing
    arrives: it must come back with MOE_ERR_DEVICE_TIMEOUT in the status word, and the next call must work."""
    inp = make_gqa_inputs(dict(B=2, Hq=32, Hkv=4, D=128, page_size=16, lengths=[5000, 300]), seed=3, device="cuda")
    ws = moe.alloc_workspace(moe.gqa_decode_workspace_bytes(2, 32, 4, 128, 5000), "cuda")
    moe.gqa_selftest_wait_timeout(ws)
    assert moe.moe_last_status(ws) == -7
    assert ws[:12].view(torch.int32)[1].item() == 12          # the site recorded next to the status
    check(inp)
    out = torch.empty((2, 32, 128), dtype=torch.bfloat16, device="cuda")
    moe.gqa_paged_decode(inp["q"], inp["k_cache"], inp["v_cache"], inp["kv_indptr"], inp["kv_indices"],
                         inp["kv_last_page_len"], 5000, inp["sm_scale"], out, ws)
    assert moe.moe_last_status(ws) == 0


def test_warps_of_a_block_whose_wait_ran_out_leave_together():
    """One warp's wait runs out while the other three have what they waited for: all four come to the answer that the
    block has no result to store.  (What three of four warps have would overwrite out with an incomplete sum.)"""
    ws = moe.alloc_workspace(256, "cuda")
    moe.gqa_selftest_wait_timeout(ws)
    assert moe.moe_last_status(ws) == -7
    assert ws[:16].view(torch.int32)[3].item() == 4


def test_a_sequence_longer_than_the_hint_is_still_computed_in_full():
    inp = make_gqa_inputs(dict(B=2, Hq=32, Hkv=4, D=128, page_size=16, lengths=[3000, 500]), seed=2, device="cuda")
    check(inp, max_kv_len=1024)     # the last split runs to the end of the sequence


def _rewritten_inputs(B, Hq, Hkv, P, length):
    """A decode call whose every input is written by kernels before each pass (256 pages): the passes' sources, what writes one
    into the buffers on the current stream (the page table by the library's router, whose kernel lets the next one start
    early), and the call."""
    pages, n = 256, B * -(-length // P)
    g = torch.Generator(device="cuda").manual_seed(B + P)
    bf16 = lambda *shape: torch.randn(*shape, generator=g, device="cuda").to(torch.bfloat16)
    sources = []
    for i in range(3):
        table = torch.randint(pages, (n,), generator=g, device="cuda")
        last = torch.randint(1, P + 1, (B,), generator=g, device="cuda", dtype=torch.int32)
        sources.append(dict(k=bf16(pages, P, Hkv, 128), v=bf16(pages, P, Hkv, 128), q=bf16(B, Hq, 128), last=last, table=table,
                            logits=torch.nn.functional.one_hot(table, pages).float()))
    k, v, q, last = (torch.zeros_like(sources[0][name]) for name in ("k", "v", "q", "last"))
    indptr = torch.arange(B + 1, dtype=torch.int32, device="cuda") * (n // B)
    ids, w = torch.zeros((n, 1), dtype=torch.int32, device="cuda"), torch.empty((n, 1), device="cuda")
    offsets, order = torch.empty(pages + 1, dtype=torch.int32, device="cuda"), torch.empty((2, n), dtype=torch.int32, device="cuda")
    route_ws = moe.alloc_workspace(moe.moe_route_workspace_bytes(n, pages, 1), "cuda")
    def write(src, last_writer):
        s = torch.cuda.current_stream()
        writers = [lambda: torch.add(src["last"], 0, out=last),
                   lambda: torch.mul(src["q"], 1, out=q),
                   lambda: torch.mul(src["v"], 1, out=v),
                   lambda: torch.mul(src["k"], 1, out=k),
                   lambda: moe.moe_route(src["logits"], 1, ids, w, offsets, order[0], order[1], route_ws, stream=s)]
        for i in range(len(writers)):
            writers[(i + last_writer + 1) % len(writers)]()
    def call(out, ws):
        moe.gqa_paged_decode(q, k, v, indptr, ids.view(-1), last, length, 0.09, out, ws, stream=torch.cuda.current_stream())
    nbytes = moe.gqa_decode_workspace_bytes(B, Hq, Hkv, 128, length)
    refs = []
    for src in sources:   # nothing overlaps
        refs.append(torch.empty_like(q))
        write(src, 0)
        torch.cuda.synchronize()
        assert torch.equal(ids.view(-1).long(), src["table"])
        ws = moe.alloc_workspace(nbytes, "cuda")
        call(refs[-1], ws)
        assert moe.moe_last_status(ws) == 0
    assert not torch.equal(refs[0], refs[1]) and not torch.equal(refs[1], refs[2])
    return sources, write, call, refs, nbytes


# the launch forms of a call that splits nothing, by blocks and tokens: on SMs of their own, short ones, a full machine,
# and in between (not started early); the row gather's the same; and a call with parts
REWRITTEN = [(3, 32, 4, 16, 400), (24, 32, 4, 16, 250), (80, 32, 4, 16, 100), (25, 32, 4, 16, 640), (3, 32, 4, 12, 300),
             (24, 32, 4, 12, 120), (120, 32, 4, 1, 8), (20, 32, 4, 12, 480), (2, 32, 4, 16, 8000)]


@pytest.mark.parametrize("B,Hq,Hkv,P,length", REWRITTEN)
def test_inputs_written_by_the_kernels_directly_in_front(B, Hq, Hkv, P, length):
    """Every input anew before every pass, each of them by the kernel directly in front of the call in turn, all queued before
    the first one runs: no pass sees what an input held before."""
    sources, write, call, refs, nbytes = _rewritten_inputs(B, Hq, Hkv, P, length)
    ws = moe.alloc_workspace(nbytes, "cuda")
    outs = [torch.empty_like(refs[0]) for _ in range(30)]
    torch.cuda.synchronize()
    torch.cuda._sleep(40_000_000)
    for i, out in enumerate(outs):
        write(sources[i % 3], i % 5)
        call(out, ws)
    assert moe.moe_last_status(ws) == 0
    for i, out in enumerate(outs):
        assert torch.equal(out.view(torch.int16), refs[i % 3].view(torch.int16)), i


@pytest.mark.parametrize("B,Hq,Hkv,P,length", REWRITTEN[:2] + REWRITTEN[4:5] + REWRITTEN[-1:])
def test_a_captured_call_behind_joined_streams_reads_what_both_wrote(B, Hq, Hkv, P, length):
    """Captured behind a fork and a join (two nodes in front), and behind a kernel that lets it start early."""
    sources, write, call, refs, nbytes = _rewritten_inputs(B, Hq, Hkv, P, length)
    ws = moe.alloc_workspace(nbytes, "cuda")
    outs = [torch.empty_like(refs[0]) for _ in range(2)]
    src = {name: t.clone() for name, t in sources[0].items()}
    fork, s = torch.cuda.Stream(), torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        fork.wait_stream(torch.cuda.current_stream())
        write(src, 0)
        with torch.cuda.stream(fork):
            scratch = src["q"] + 1
        torch.cuda.current_stream().wait_stream(fork)
        call(outs[0], ws)
        write(src, 4)
        call(outs[1], ws)
    for i in (1, 2, 0, 1):
        for name, t in sources[i].items():
            src[name].copy_(t)
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        assert moe.moe_last_status(ws) == 0
        for out in outs:
            assert torch.equal(out.view(torch.int16), refs[i].view(torch.int16))
    del scratch


def test_results_do_not_depend_on_which_block_finishes_last():
    inp = make_gqa_inputs(dict(B=3, Hq=32, Hkv=4, D=128, page_size=16, lengths=[9000, 4000, 12345]), seed=4, device="cuda")
    first, lse0 = run_gpu(inp)
    for _ in range(5):
        again, lse1 = run_gpu(inp)
        assert torch.equal(first.view(torch.int16), again.view(torch.int16)) and torch.equal(lse0, lse1)


def test_lse_is_optional_and_arguments_are_checked_before_any_launch():
    inp = make_gqa_inputs("gqa_tiny", seed=0, device="cuda")
    out, _ = run_gpu(inp, want_lse=False)
    ref, _ = oracle(inp)
    assert (np.abs(out.float().cpu().numpy() - ref) <= OUT_TOL * (1 + np.abs(ref))).all()
    B, Hq, Hkv, D = inp["B"], inp["Hq"], inp["Hkv"], inp["D"]
    ws = moe.alloc_workspace(moe.gqa_decode_workspace_bytes(B, Hq, Hkv, D, 70), "cuda")
    o = torch.zeros((B, Hq, D), dtype=torch.bfloat16, device="cuda")
    args = (inp["q"], inp["k_cache"], inp["v_cache"], inp["kv_indptr"], inp["kv_indices"], inp["kv_last_page_len"])
    assert moe.gqa_paged_decode(*args, 70, 0.1, o, ws[:256], check=False) == -5            # workspace too small
    assert moe.gqa_paged_decode(*args, 70, 0.1, o, ws[8:], check=False) == -4              # workspace misaligned
    bad_q = torch.zeros((B, 7, D), dtype=torch.bfloat16, device="cuda")                     # 7 heads over 2 kv heads
    assert moe.gqa_paged_decode(bad_q, *args[1:], 70, 0.1, o, ws, check=False) == -3
    assert moe.gqa_decode_workspace_bytes(B, Hq, Hkv, 64, 70) == 0                          # D must be 128
    torch.cuda.synchronize()
    assert (o == 0).all()


@pytest.mark.parametrize("name", ["gqa_decode_b64", "gqa_decode_b256", "gqa_decode_b1_long", "gqa_decode_b64_16k"])
def test_full_size_workload(name):
    """The benchmark's workloads in its launch configuration: every element against the oracle."""
    inp = make_gqa_inputs(GQA_CONFIGS[name], seed=0, device="cuda")
    out = check(inp)
    again, _ = run_gpu(inp)
    assert torch.equal(out.view(torch.int16), again.view(torch.int16))
