"""GPU parity: the CUDA prune step, called through the C ABI, against the CPU oracle on the
same seeded inputs.  Sizes span several 128-wide tiles with ragged tails; the benchmark shapes
run at full size with the oracle evaluated on a sample of the sequences."""
import math

import numpy as np
import pytest
import torch

from paper_2603_14549_b200 import binding as A
from paper_2603_14549_b200 import workloads as W
from tests.parity import check_invariants, compare_sample

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    c = A.asap_init(0, max_total_tokens=80000, max_B=32, max_H=40, max_D=5120, max_keep_rows=40000)
    yield c
    A.asap_free(c)


def run_step(ctx, batch, params, rank_start=None, rank_len=None, samples=None, stats=None):
    inp = A.make_inputs(batch, DEV, rank_start, rank_len)
    out = A.alloc_outputs(inp, params.keep_k, fill=True, per_head=params.per_head_mask)
    A.asap_prune_step(ctx, inp, params, out)
    torch.cuda.synchronize()
    A.asap_check(ctx)
    for b in (range(batch.B) if samples is None else samples):
        compare_sample(batch, b, params, out, rank_start, rank_len, stats)
    if samples is not None:          # the oracle saw a sample of the batch: every sequence still has to be well formed
        for b in range(batch.B):
            check_invariants(batch, b, params, out)
    return inp, out


def test_ragged_multi_tile(ctx):
    batch = W.tiny(B=3, n_vis=[130, 257, 64], text_lens=[5, 17, 33], H=2, keep_k=16, seed=101, centres=6)
    run_step(ctx, batch, A.Params(keep_k=16))


@pytest.mark.parametrize("k", [300, 512, 257])
def test_two_slot_tiles_in_one_pass(ctx, k):
    """257 .. 512 kept slots: two groups of slots, dealt to neighbouring blocks of two row tiles each, one pass over the hidden
    dimension (300 and 257 leave a ragged second group, 512 fills every column)."""
    batch = W.tiny(B=2, n_vis=[700, 650], text_lens=[12, 40], H=2, keep_k=k, seed=107, centres=30)
    run_step(ctx, batch, A.Params(keep_k=k))


@pytest.mark.parametrize("nvs,texts,H", [([128, 129, 9], [240, 241, 500], 2), ([64, 300, 20] * 14, [5, 250, 1] * 14, 8)],
                         ids=["tile_edges", "many_items_per_block"])
def test_query_sums_inside_the_score_kernel(ctx, nvs, texts, H):
    """The visual queries are added up beside the key tiles: spans that end on a tile edge, one past it and inside
    the first tile; ranking rows of one, two and three row pairs (only the first carries the masses); and more
    (sequence, head) items than blocks, so that ring positions run on from one item to the next."""
    batch = W.tiny(B=len(nvs), n_vis=nvs, text_lens=texts, H=H, keep_k=8, seed=140 + H, centres=6)
    big = A.asap_init(0, max_total_tokens=batch.total + len(nvs) * 300, max_B=len(nvs), max_H=H, max_D=H * 128)
    try:
        run_step(big, batch, A.Params(keep_k=8), samples=range(len(nvs)) if len(nvs) < 4 else [0, 1, 2, len(nvs) - 1])
    finally:
        A.asap_free(big)


@pytest.mark.parametrize("B,H,skipped,visual", [
    (64, 4, [], 0),                    # 256 items, the most sequences that are drawn by size; the first round ends with a sequence
    (65, 4, [0, 64], 0),               # one sequence more: drawn in order
    (60, 5, [0, 1, 2, 29, 30, 59], 0), # the first round ends inside sequence 29, which is skipped
    (37, 12, [11, 12, 13], 0),         # inside sequence 12; three rounds
    (11, 40, [0, 3, 10], 0),           # inside sequence 3
    (60, 5, list(range(31)), 0),       # every item of the first round is skipped
    (60, 5, [0, 1, 2, 29, 30, 59], 2), # masses in front, at most four tiles per item: the ring takes several items at once
], ids=["most", "one_more", "skipped", "rounds", "wide", "first_round_skipped", "rows"])
def test_items_drawn_by_size(B, H, skipped, visual):
    """Image spans of different lengths in more (sequence, head) items than blocks: after the first round the items are drawn by
    size.  Each head of each sequence comes once, whichever sequences are skipped (every sequence's scores against the oracle),
    and the call repeats bit for bit."""
    nvs = [16 + (37 * b) % 150 for b in range(B)]
    batch = W.tiny(B=B, n_vis=nvs, text_lens=[3 + (11 * b) % 40 for b in range(B)], H=H, keep_k=8, seed=370 + B, centres=5)
    rank = (batch.text_start - visual, batch.text_len + visual) if visual else (None, None)
    inp = A.make_inputs(batch, DEV, *rank)
    for b in skipped:
        inp.text_len[b] = 9999
        if visual:
            inp.rank_len[b] = 9999
    p = A.Params(keep_k=8)
    c = A.asap_init(0, max_total_tokens=batch.total + B * 166, max_B=B, max_H=H, max_D=H * 128)
    try:
        outs = []
        for _ in range(20):
            out = A.alloc_outputs(inp, 8, fill=True)
            A.asap_prune_step(c, inp, p, out)
            torch.cuda.synchronize()
            if skipped:
                with pytest.raises(A.AsapError) as e:
                    A.asap_check(c)
                assert e.value.status == -6 and "timed out" not in str(e.value)
            else:
                A.asap_check(c)
            outs.append(out)
    finally:
        A.asap_free(c)
    valid = [b for b in range(B) if b not in skipped]
    for out in outs[1:]:
        for f in ("mass", "salience", "rank_score", "keep_idx", "assign", "out_hidden"):
            assert torch.equal(getattr(out, f), getattr(outs[0], f)), f
    for b in valid:
        compare_sample(batch, b, p, outs[0], *rank)
    assert not skipped or float(outs[0].rank_score[skipped].abs().max()) == 0.0


def test_items_drawn_by_size_on_two_streams():
    """Two contexts whose score kernels contend for the SMs: blocks of the second start one by one as blocks of the first leave, some
    only when the others have drawn all items of the first rounds.  Every result is that of the call by itself."""
    B, H = 40, 8
    batches, inps, ctxs, want = [], [], [], []
    p = A.Params(keep_k=12)
    for i in range(2):
        nvs = [20 + (53 * b + 300 * i * (b % 3)) % 700 for b in range(B)]
        batches.append(W.tiny(B=B, n_vis=nvs, text_lens=[4 + (b * 7) % 90 for b in range(B)], H=H, keep_k=12, seed=380 + i, centres=5))
        inps.append(A.make_inputs(batches[i], DEV))
    streams = [torch.cuda.Stream() for _ in range(2)]
    for i in range(2):
        ctxs.append(A.asap_init(0, max_total_tokens=batches[i].total + B * 720, max_B=B, max_H=H, max_D=H * 128))
    try:
        for i in range(2):
            out = A.alloc_outputs(inps[i], 12, fill=True)
            A.asap_prune_step(ctxs[i], inps[i], p, out)
            torch.cuda.synchronize()
            A.asap_check(ctxs[i])
            want.append(out)
        outs = [[A.alloc_outputs(inps[i], 12, fill=True) for _ in range(16)] for i in range(2)]
        torch.cuda.synchronize()
        for n in range(16):
            for i in range(2):
                A.asap_prune_step(ctxs[i], inps[i], p, outs[i][n], streams[i])
        torch.cuda.synchronize()
        for i in range(2):
            A.asap_check(ctxs[i], streams[i])
            for out in outs[i]:
                for f in ("mass", "salience", "rank_score", "keep_idx", "drop_idx", "assign", "out_hidden", "out_pos", "src_row"):
                    n = int(want[i].out_cu_seqlens[-1]) if f in ("out_hidden", "out_pos", "src_row") else None
                    assert torch.equal(getattr(out, f)[:n], getattr(want[i], f)[:n]), f
    finally:
        for c in ctxs:
            A.asap_free(c)


@pytest.mark.parametrize("per_head,visual", [(False, 0), (False, 5), (True, 0), (True, 5)], ids=["text", "rows", "heads", "heads_rows"])
@pytest.mark.parametrize("text", [3, 37, 127, 128, 245, 491])
def test_a_sequence_does_not_see_its_neighbours(ctx, text, per_head, visual):
    """Everything of the next sequence is NaN or infinite (query rows up to the next multiple of 16 are multiplied with a
    sequence's last ranking rows, key and hidden rows lie in its last tiles): not one bit of the sequence's results changes."""
    batch = W.tiny(B=2, n_vis=[150, 140], text_lens=[text, 9], H=2, keep_k=30, seed=619, centres=6)
    rank = (batch.text_start - visual, batch.text_len + visual) if visual else (None, None)
    p = A.Params(keep_k=30, per_head_mask=per_head)
    outs = []
    for spoil in (False, True):
        if spoil:
            bad = torch.tensor([float("nan"), float("inf"), -float("inf")], dtype=torch.bfloat16)
            rows = torch.arange(int(batch.cu_seqlens[1]), batch.total)
            for i, t in enumerate((batch.q, batch.k, batch.hidden)):
                t[rows] = bad[(rows + i) % 3].reshape(-1, *([1] * (t.dim() - 1)))
        inp = A.make_inputs(batch, DEV, *rank)
        out = A.alloc_outputs(inp, 30, fill=True, per_head=per_head)
        A.asap_prune_step(ctx, inp, p, out)
        score = A.alloc_outputs(inp, 30, fill=True, per_head=per_head)
        A.asap_score(ctx, inp, p, score)
        torch.cuda.synchronize()
        A.asap_check(ctx)
        outs.append((out, score))
    n = int(outs[0][0].out_cu_seqlens[1])
    for good, bad in zip(*outs):
        for f in ("mass", "salience", "mask_log", "rank_score", "keep_idx", "drop_idx", "assign", "best_sim", "mask_log_heads"):
            if getattr(good, f) is not None and (good is outs[0][0] or f in ("mass", "salience", "rank_score")):
                assert torch.equal(getattr(good, f)[0], getattr(bad, f)[0]), f
    for f in ("out_hidden", "out_pos", "src_row"):
        assert torch.equal(getattr(outs[0][0], f)[:n], getattr(outs[1][0], f)[:n]), f


@pytest.mark.parametrize("H", [16, 20, 32, 40])
@pytest.mark.parametrize("nvs", [[576], [1201, 1204, 300]], ids=["one", "ragged"])
def test_masses_in_the_score_kernel_lose_no_precision(ctx, nvs, H):
    """Eq. 1 from the tensor cores against 64 bits, heads of either sign.  The rounding of the result alone is 2^-24 / sqrt(3) =
    3.4e-8 (2-norm); separate fp32 kernels for query sum and masses are off by 1.04e-7 to 1.33e-7 on these batches, and one
    accumulator that all k-steps of a head add to by 1.26e-7 to 1.75e-7."""
    batch = W.tiny(B=len(nvs), n_vis=nvs, text_lens=[9 + b for b in range(len(nvs))], H=H, keep_k=40, seed=160 + H, centres=9)
    inp = A.make_inputs(batch, DEV)
    out = A.alloc_outputs(inp, 40, fill=True)
    A.asap_prune_step(ctx, inp, A.Params(keep_k=40), out)
    torch.cuda.synchronize()
    A.asap_check(ctx)
    err = tot = 0.0
    for b, nv in enumerate(nvs):
        lo = int(batch.cu_seqlens[b]) + int(batch.vis_start[b])
        q, k = inp.q[lo:lo + nv].double(), inp.k[lo:lo + nv].double()
        s = (k * q.sum(0)).sum((1, 2)) / (H * math.sqrt(128))
        err += float(((out.mass[b, :nv].double() - s) ** 2).sum())
        tot += float((s ** 2).sum())
    print("mass error, 2-norm:", math.sqrt(err / tot))
    assert math.sqrt(err / tot) < 1.04e-7


@pytest.mark.parametrize("nvs,k", [([65, 66], 1), ([129, 130, 32, 33], 1), ([4096, 4097, 4129], 1), ([1028, 1029], 4), ([2500, 1030], 3),
                                   ([40, 16], 16), ([2060], 7)],
                         ids=["a_full_list", "two_lists_and_word_edges", "a_full_pass", "words_of_few", "several_lists", "nothing_dropped", "one"])
def test_few_slots_with_many_members(ctx, nvs, k):
    """A slot's members come from its row of bits, 32 visual tokens a word, 4096 a pass, and are merged 64 at a time.  With one slot
    everything else is its member: 64 and 65, 128 and 129 members, spans that end on a word or one past it, on a pass, one and 33 past it;
    a sequence without a dropped token."""
    batch = W.tiny(B=len(nvs), n_vis=nvs, text_lens=[9 + b for b in range(len(nvs))], H=2, keep_k=k, seed=120 + k, centres=k + 1)
    run_step(ctx, batch, A.Params(keep_k=k))


@pytest.mark.parametrize("nvs,k,tokens", [([4200, 33], 20, 9000), ([4097, 64], 16, 9000), ([640, 610], 310, 1400)],
                         ids=["two_passes_long_lists", "one_member_past_a_pass", "grouped_instead"])
def test_rows_of_member_bits(nvs, k, tokens):
    """A slot's members as a row of bits: more words than a warp takes per pass (4096 tokens), more members than its list holds
    (64), a sequence whose last token alone lies in the second pass, and a context (310 kept slots, width 256, few tokens) whose
    scratch has no room for the rows, so that the similarity kernel groups the members."""
    batch = W.tiny(B=len(nvs), n_vis=nvs, text_lens=[9 + b for b in range(len(nvs))], H=2, keep_k=k, seed=310 + k, centres=11)
    small = A.asap_init(0, max_total_tokens=tokens, max_B=len(nvs), max_H=2, max_D=256)
    try:
        run_step(small, batch, A.Params(keep_k=k))
    finally:
        A.asap_free(small)


@pytest.mark.parametrize("k", [680, 700], ids=["bits", "grouped"])
def test_long_rows_of_member_bits(ctx, k):
    """Rows of bits in two passes: from some 690 slots of eight sequences of 4224 tokens on (148 SMs) the members are grouped instead."""
    batch = W.tiny(B=8, n_vis=[4224] + [4000 - 100 * b for b in range(7)], text_lens=[4 + b for b in range(8)], H=1, keep_k=k, seed=341, centres=90)
    run_step(ctx, batch, A.Params(keep_k=k), samples=[0, 7])


@pytest.mark.parametrize("nv", [576, 577], ids=["eight_rows_a_block", "one_more_member"])
def test_grouped_members_of_many_slots(nv):
    """Width 128 has no room for the bits of 192 kept slots: grouped members, up to two a slot on average with eight slots per block,
    beyond that with one."""
    batch = W.tiny(B=13, n_vis=[nv] + [576 - 20 * b for b in range(12)], text_lens=[4 + b for b in range(13)], H=1, keep_k=192, seed=340, centres=40)
    c = A.asap_init(0, max_total_tokens=13 * 592, max_B=13, max_H=1, max_D=128)
    try:
        run_step(c, batch, A.Params(keep_k=192))
    finally:
        A.asap_free(c)


@pytest.mark.parametrize("k,H", [(600, 1), (600, 3), (340, 5), (1100, 1)], ids=["fewer_steps_than_groups", "two_steps_each", "uneven", "five_groups"])
def test_row_norms_shared_by_the_groups(ctx, k, H):
    """Every group of kept slots adds up the squares of its range of the columns: two 64-column steps for three or five groups (some
    have none), and ranges of different lengths; pairs of row tiles whose second tile is empty or holds one row."""
    batch = W.tiny(B=2, n_vis=[1300, 1409], text_lens=[12, 30], H=H, keep_k=k, seed=330 + H, centres=50)
    run_step(ctx, batch, A.Params(keep_k=k))


@pytest.mark.parametrize("per_head", [False, True], ids=["mean", "heads"])
@pytest.mark.parametrize("nvs,H", [([127, 128, 129, 641], 2), ([40, 300, 90, 256] * 10, 4)], ids=["tile_edges", "many_items_per_block"])
def test_masses_with_visual_ranking_rows(nvs, H, per_head):
    """The mass kernel streams a head's queries, then its keys, 128 rows a tile: spans that end on a tile edge and beside it, and more
    (sequence, head) items than blocks, so that the ring runs on from one item to the next."""
    B = len(nvs)
    batch = W.tiny(B=B, n_vis=nvs, text_lens=[5 + b % 7 for b in range(B)], H=H, keep_k=24, seed=350 + B, centres=6)
    big = A.asap_init(0, max_total_tokens=batch.total + B * 641, max_B=B, max_H=H, max_D=H * 128)
    try:
        run_step(big, batch, A.Params(keep_k=24, per_head_mask=per_head, lambda_max=0.7), batch.text_start - 9, batch.text_len + 9,
                 samples=range(B) if B < 5 else [0, 1, 2, B - 2, B - 1])
    finally:
        A.asap_free(big)


def test_many_row_tiles_and_three_slot_tiles(ctx):
    """A batch large enough that the similarity kernel runs unsliced with more blocks than SMs
    (15 sequences x 19 row tiles) and three slot tiles (600 kept slots).  Odd and even numbers of row
    tiles, a ragged last tile of one row; the oracle checks three sequences."""
    nvs = [2350 if b % 2 else 2432 for b in range(15)]
    nvs[0] = 2305                                               # 19 row tiles, one row in the last
    batch = W.tiny(B=15, n_vis=nvs, text_lens=[6 + b for b in range(15)], H=2, keep_k=600, seed=108, centres=40)
    run_step(ctx, batch, A.Params(keep_k=600), samples=[0, 1, 14])


def test_a_late_dominant_key_moves_the_softmax_reference(ctx):
    """One visual key far into the sequence is scaled so that its logits exceed every earlier logit of a
    ranking row by hundreds of nats (or fall that far below, for rows whose dot product is negative).  A
    running sum kept relative to an early maximum would overflow there: the row's reference has to move,
    and the probabilities of all other keys have to come out as (correctly) vanishing."""
    batch = W.tiny(B=2, n_vis=[400, 330], text_lens=[40, 150], H=2, keep_k=50, seed=110, centres=8)
    for b, where in ((0, 300), (1, 200)):
        row = int(batch.cu_seqlens[b]) + int(batch.vis_start[b]) + where
        batch.k[row] = (batch.k[row].float() * 300.0).to(torch.bfloat16)
    run_step(ctx, batch, A.Params(keep_k=50))


def test_text_longer_than_one_row_tile(ctx):
    batch = W.tiny(B=2, n_vis=[200, 140], text_lens=[150, 129], H=2, keep_k=40, seed=102, centres=8)
    run_step(ctx, batch, A.Params(keep_k=40))


@pytest.mark.parametrize("lambda_max", [1.0, 0.5, 0.1])
def test_visual_ranking_rows_use_the_soft_mask(ctx, lambda_max):
    batch = W.tiny(B=2, n_vis=[300, 129], text_lens=[20, 7], H=2, keep_k=32, seed=103, centres=8)
    rs = batch.vis_start.clone()
    rl = batch.vis_len + batch.text_len            # ranking rows = image span + text span
    run_step(ctx, batch, A.Params(keep_k=32, lambda_max=lambda_max), rs, rl)


@pytest.mark.parametrize("lambda_max", [1.0, 0.3])
def test_per_head_masks_with_visual_ranking_rows(ctx, lambda_max):
    """Eq. 1-3 per head: four heads with their own salience and mask vector; the ranking rows include
    the image span, so every head's logits are really shifted by that head's mask."""
    batch = W.tiny(B=2, n_vis=[300, 129], text_lens=[20, 7], H=4, keep_k=32, seed=105, centres=8)
    rs = batch.vis_start.clone()
    rl = batch.vis_len + batch.text_len
    inp, out = run_step(ctx, batch, A.Params(keep_k=32, lambda_max=lambda_max, per_head_mask=True), rs, rl)
    mh = out.mask_log_heads.cpu()
    assert float((mh[0, 0, :300] - mh[0, 1, :300]).abs().max()) > 1e-3      # the heads' masks do differ


def test_per_head_masks_with_text_ranking_rows(ctx):
    batch = W.tiny(B=3, n_vis=[130, 257, 64], text_lens=[5, 17, 33], H=2, keep_k=16, seed=106, centres=6)
    run_step(ctx, batch, A.Params(keep_k=16, per_head_mask=True))


def test_ranking_rows_partly_visual_and_mask_off(ctx):
    batch = W.tiny(B=2, n_vis=[260, 131], text_lens=[9, 30], H=1, keep_k=20, seed=104)
    rs = batch.vis_start + 100
    rl = batch.vis_len - 100 + batch.text_len
    run_step(ctx, batch, A.Params(keep_k=20, lambda_max=0.7), rs, rl)
    run_step(ctx, batch, A.Params(keep_k=20, mask_enable=False), rs, rl)


def test_identity_when_k_equals_visual_count(ctx):
    batch = W.tiny(B=2, n_vis=[150, 150], text_lens=[4, 40], H=2, keep_k=150, seed=105)
    inp, out = run_step(ctx, batch, A.Params(keep_k=150))
    assert torch.equal(out.out_hidden.cpu(), batch.hidden)
    assert torch.equal(out.out_pos.cpu(), batch.pos_ids)


def test_one_sequence_keeps_everything_while_another_merges(ctx):
    """keep_k equals the first sequence's visual count (nothing dropped there, its rows are copies) while
    the second one drops and merges 80 tokens."""
    batch = W.tiny(B=2, n_vis=[150, 230], text_lens=[9, 21], H=2, keep_k=150, seed=109, centres=9)
    inp, out = run_step(ctx, batch, A.Params(keep_k=150))
    n0 = int(batch.cu_seqlens[1])
    assert torch.equal(out.out_hidden[:n0].cpu(), batch.hidden[:n0])
    assert int((out.assign[0] >= 0).sum()) == 0 and int((out.assign[1] >= 0).sum()) == 80


def test_mask_off_merge_off_is_plain_topk_gather(ctx):
    batch = W.tiny(B=2, n_vis=[190, 133], text_lens=[12, 31], H=2, keep_k=24, seed=106)
    inp, out = run_step(ctx, batch, A.Params(keep_k=24, mask_enable=False, merge_enable=False))
    n_out = int(out.out_cu_seqlens[-1])                 # the buffers are sized for the worst case
    src = out.src_row[:n_out].cpu().long()
    assert torch.equal(out.out_hidden[:n_out].cpu(), batch.hidden[src])


@pytest.mark.parametrize("t", [0.8, 0.95, 1.0])
def test_similarity_threshold(ctx, t):
    batch = W.tiny(B=2, n_vis=[180, 140], text_lens=[10, 20], H=2, keep_k=30, seed=107, centres=5)
    inp, out = run_step(ctx, batch, A.Params(keep_k=30, sim_threshold=t))
    if t >= 1.0:
        assert int((out.assign >= 0).sum()) == 0


@pytest.mark.parametrize("nv", [1, 2, 3, 5, 8, 127, 128, 129])
@pytest.mark.parametrize("tl", [1, 16, 17])
def test_edge_sizes(ctx, nv, tl):
    ks = sorted({1, max(1, nv - 1), nv})
    for k in ks:
        batch = W.tiny(B=2, n_vis=[nv, nv], text_lens=[tl, tl + 1], H=1, keep_k=k, seed=200 + nv, centres=2)
        run_step(ctx, batch, A.Params(keep_k=k))


def test_duplicate_token_merges_into_its_twin(ctx):
    """Ranking reads only Q and K, so overwriting a dropped token's hidden row does not change the kept
    set: the token stays dropped, and as a copy of a kept row it must land on that row's slot with
    similarity 1 (no other kept row equals it: the rows are noisy draws)."""
    batch = W.tiny(B=1, n_vis=[140], text_lens=[8], H=2, keep_k=20, seed=108, centres=50)
    inp = A.make_inputs(batch, DEV)
    out = A.alloc_outputs(inp, 20, fill=True)
    p = A.Params(keep_k=20)
    A.asap_prune_step(ctx, inp, p, out)
    torch.cuda.synchronize()
    keep = out.keep_idx[0].cpu()
    drop = out.drop_idx[0].cpu()
    v0 = int(batch.vis_start[0])
    victim = int(drop[5])
    batch.hidden[v0 + victim] = batch.hidden[v0 + int(keep[3])]
    inp2, out2 = run_step(ctx, batch, p)
    assert torch.equal(out2.keep_idx[0].cpu(), keep)          # same Q / K, same ranking
    pos = (out2.drop_idx[0] == victim).nonzero()
    assert len(pos) == 1
    dp = int(pos[0])
    assert int(out2.assign[0, dp]) == 3
    assert abs(float(out2.best_sim[0, dp]) - 1.0) < 1e-5


def test_c1_full(ctx):
    stats = {}
    batch = W.config("c1")
    run_step(ctx, batch, A.Params(keep_k=batch.keep_k), stats=stats)
    print("c1 parity maxima", stats)


def test_c2_full_size_sampled(ctx):
    stats = {}
    batch = W.config("c2")
    run_step(ctx, batch, A.Params(keep_k=batch.keep_k), samples=[0, 7, 15], stats=stats)
    print("c2 parity maxima", stats)


@pytest.mark.parametrize("k", [320, 160])
def test_c3_prefix_with_outliers(ctx, k):
    stats = {}
    batch = W.config("c3", B=2, keep_k=k)
    run_step(ctx, batch, A.Params(keep_k=k), samples=[1], stats=stats)
    print("c3 parity maxima", stats)


def test_c4_prefix_sampled(ctx):
    stats = {}
    batch = W.config("c4", B=6)
    run_step(ctx, batch, A.Params(keep_k=batch.keep_k), samples=[5], stats=stats)
    print("c4 parity maxima", stats)


@pytest.fixture(scope="module")
def big_ctx():
    """Capacity of the largest benchmark shape (64 sequences of 35 + 2880 + up to 256 tokens)."""
    c = A.asap_init(0, max_total_tokens=64 * (35 + 2880 + 256), max_B=64, max_H=40, max_D=5120,
                    max_keep_rows=64 * 1152)
    yield c
    A.asap_free(c)


@pytest.mark.parametrize("k", [320, 160])
def test_c3_full_size_sampled(big_ctx, k):
    """The whole LLaVA-NeXT batch of 8 as bench.py runs it; the oracle checks two sequences."""
    stats = {}
    batch = W.config("c3", keep_k=k)
    run_step(big_ctx, batch, A.Params(keep_k=k), samples=[0, 7], stats=stats)
    print("c3 full parity maxima", stats)


@pytest.mark.parametrize("k", [510, 340])
def test_c6_internvl_shape_full_size_sampled(big_ctx, k):
    """InternVL-2.5-8B-shaped batch (1536 visual tokens in six tiles of 256) at the two budgets of
    Sec. 5.4 (~510 and ~340 tokens); neither is a multiple of 16, so the similarity kernel's kept-slot
    tiles are ragged.  The oracle checks two sequences."""
    stats = {}
    batch = W.config("c6", keep_k=k)
    run_step(big_ctx, batch, A.Params(keep_k=k), samples=[0, 7], stats=stats)
    print("c6 full parity maxima", stats)


def test_c4_full_size_sampled(big_ctx):
    """The AnyRes throughput shape at full size (64 sequences, 2880 visual tokens, ragged text up
    to 256 rows = two ranking-row tiles); the oracle checks the first and the last sequence."""
    stats = {}
    batch = W.config("c4")
    run_step(big_ctx, batch, A.Params(keep_k=batch.keep_k), samples=[0, 63], stats=stats)
    print("c4 full parity maxima", stats)


def test_c5_full_size_first_step_sampled(big_ctx):
    """13B-shaped batch of 32 (D = 5120, 40 heads), first step 2304 -> 1152, at full size."""
    stats = {}
    batch = W.config("c5")
    run_step(big_ctx, batch, A.Params(keep_k=batch.keep_k), samples=[31], stats=stats)
    print("c5 full parity maxima", stats)


def _c5_schedule(ctx, B, samples):
    batch = W.config("c5", B=B)
    cur = batch
    for step, k in enumerate(W.C5_SCHEDULE):
        p = A.Params(keep_k=k)
        cur.keep_k = k
        stats = {}
        inp, out = run_step(ctx, cur, p, samples=samples, stats=stats)
        print(f"c5 step {step + 1} (B = {B}) parity maxima", stats)
        ocu = out.out_cu_seqlens.cpu()
        hidden = out.out_hidden[: int(ocu[-1])].cpu()
        pos = out.out_pos[: int(ocu[-1])].cpu()
        q, kk = W.redraw_qk(pos, ocu, cur.H, cur.head_dim, cur.seed, step + 1)
        cur = W.Batch(name="c5", B=cur.B, H=cur.H, head_dim=cur.head_dim, D=cur.D, keep_k=k, cu_seqlens=ocu,
                      vis_start=cur.vis_start, vis_len=torch.full_like(cur.vis_len, k),
                      text_start=cur.vis_start + k, text_len=cur.text_len, q=q, k=kk, hidden=hidden,
                      pos_ids=pos, seed=cur.seed)


def test_c5_progressive_three_steps(ctx):
    """13B-shaped schedule 2304 -> 1152 -> 576 -> 288: every step consumes the previous step's
    hidden states and gathered position ids, with Q/K re-drawn at those positions."""
    _c5_schedule(ctx, 2, [1])


def test_c5_progressive_three_steps_full_batch(big_ctx):
    """The same schedule on the whole batch of 32 (the sizes the benchmark times): the oracle checks one
    sequence per step, every other sequence is checked for the properties that need no oracle."""
    _c5_schedule(big_ctx, 32, [17])
