"""The give-up path of the bounded waits in the three tensor-core kernels, exercised in the harmless
form: the wait limit of ONE call is set to a single clock cycle, so a healthy run gives up at its
first wait that is not satisfied at once.  The call must return, asap_check must name the kernel's
time-out bit, and the next ordinary call on the same context must give the results of a fresh one
bit for bit.  Nothing is made to hang and nothing is expected to fault: the blocks leave through
the same teardown as always, after draining the copies and MMAs they have in flight."""
import pytest
import torch

from paper_2603_14549_b200 import binding as A
from paper_2603_14549_b200 import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    c = A.asap_init(0, max_total_tokens=20000, max_B=8, max_H=4, max_D=512, max_keep_rows=8000)
    yield c
    A.asap_free(c)


def _same(a, b, names):
    for n in names:
        x, y = getattr(a, n), getattr(b, n)
        assert torch.equal(x, y), n


def test_score_kernel_gives_up_and_the_context_recovers(ctx):
    batch = W.tiny(B=3, n_vis=[300, 260, 140], text_lens=[20, 150, 7], H=2, keep_k=40, seed=601, centres=6)
    inp = A.make_inputs(batch, DEV)
    p = A.Params(keep_k=40)
    good = A.alloc_outputs(inp, 40, fill=True)
    A.asap_prune_step(ctx, inp, p, good)
    torch.cuda.synchronize(); A.asap_check(ctx)

    bad = A.alloc_outputs(inp, 40, fill=True)
    A.asap_debug_wait_limit(ctx, 1)
    A.asap_prune_step(ctx, inp, p, bad)              # returns normally; its results are void
    torch.cuda.synchronize()
    with pytest.raises(A.AsapError) as e:
        A.asap_check(ctx)
    assert e.value.status == -6 and "timed out in the score kernel" in str(e.value)

    again = A.alloc_outputs(inp, 40, fill=True)       # the limit held for one call only
    A.asap_prune_step(ctx, inp, p, again)
    torch.cuda.synchronize(); A.asap_check(ctx)
    _same(good, again, ("rank_score", "keep_idx", "drop_idx", "assign", "out_hidden", "out_pos", "src_row", "out_cu_seqlens"))


def test_score_kernel_that_draws_by_size_gives_up_and_the_context_recovers():
    """The same where items past the first round wait for their order too (image spans of different lengths, 240 items)."""
    B = 60
    batch = W.tiny(B=B, n_vis=[30 + (41 * b) % 170 for b in range(B)], text_lens=[3 + b % 9 for b in range(B)], H=4, keep_k=10, seed=612, centres=6)
    c = A.asap_init(0, max_total_tokens=batch.total + B * 200, max_B=B, max_H=4, max_D=512)
    try:
        inp = A.make_inputs(batch, DEV)
        p = A.Params(keep_k=10)
        outs = [A.alloc_outputs(inp, 10, fill=True) for _ in range(3)]
        A.asap_prune_step(c, inp, p, outs[0])
        torch.cuda.synchronize(); A.asap_check(c)
        A.asap_debug_wait_limit(c, 1)
        A.asap_prune_step(c, inp, p, outs[1])            # returns normally; its results are void
        torch.cuda.synchronize()
        with pytest.raises(A.AsapError) as e:
            A.asap_check(c)
        assert e.value.status == -6 and "timed out in the score kernel" in str(e.value)
        A.asap_prune_step(c, inp, p, outs[2])
        torch.cuda.synchronize(); A.asap_check(c)
        _same(outs[0], outs[2], ("mass", "rank_score", "keep_idx", "drop_idx", "assign", "out_hidden", "out_pos", "src_row", "out_cu_seqlens"))
    finally:
        A.asap_free(c)


@pytest.mark.parametrize("per_head", [False, True], ids=["mean", "heads"])
def test_mass_kernel_gives_up_and_the_context_recovers(ctx, per_head):
    batch = W.tiny(B=3, n_vis=[300, 260, 140], text_lens=[20, 150, 7], H=2, keep_k=40, seed=611, centres=6)
    inp = A.make_inputs(batch, DEV, batch.text_start - 3, batch.text_len + 3)
    p = A.Params(keep_k=40, per_head_mask=per_head)
    outs = [A.alloc_outputs(inp, 40, fill=True, per_head=per_head) for _ in range(3)]
    A.asap_prune_step(ctx, inp, p, outs[0])
    torch.cuda.synchronize(); A.asap_check(ctx)
    A.asap_debug_wait_limit(ctx, 1)
    A.asap_prune_step(ctx, inp, p, outs[1])          # returns normally; its results are void
    torch.cuda.synchronize()
    with pytest.raises(A.AsapError) as e:
        A.asap_check(ctx)
    assert e.value.status == -6 and "timed out in the mass kernel" in str(e.value)
    A.asap_prune_step(ctx, inp, p, outs[2])
    torch.cuda.synchronize(); A.asap_check(ctx)
    _same(outs[0], outs[2], ("mass", "salience", "rank_score", "keep_idx", "drop_idx", "assign", "out_hidden", "out_pos", "src_row", "out_cu_seqlens"))


def test_similarity_kernel_gives_up_and_the_context_recovers(ctx):
    batch = W.tiny(B=2, n_vis=[400, 330], text_lens=[9, 12], H=2, keep_k=150, seed=602, centres=9)
    inp = A.make_inputs(batch, DEV)
    p = A.Params(keep_k=150)
    good = A.alloc_outputs(inp, 150, fill=True)
    A.asap_prune_step(ctx, inp, p, good)
    torch.cuda.synchronize(); A.asap_check(ctx)
    args = (good.salience.clone(), good.keep_idx.clone(), good.drop_idx.clone())

    ref = A.alloc_outputs(inp, 150, fill=True)
    A.asap_merge(ctx, inp, p, *args, ref)
    torch.cuda.synchronize(); A.asap_check(ctx)

    bad = A.alloc_outputs(inp, 150, fill=True)
    A.asap_debug_wait_limit(ctx, 1)
    A.asap_merge(ctx, inp, p, *args, bad)
    torch.cuda.synchronize()
    with pytest.raises(A.AsapError) as e:
        A.asap_check(ctx)
    assert e.value.status == -6 and "timed out in the similarity kernel" in str(e.value)

    again = A.alloc_outputs(inp, 150, fill=True)
    A.asap_merge(ctx, inp, p, *args, again)
    torch.cuda.synchronize(); A.asap_check(ctx)
    _same(ref, again, ("assign", "best_sim", "out_hidden", "out_pos", "src_row", "out_cu_seqlens"))


def test_gathered_similarity_gives_up_and_the_context_recovers():
    """Enough sequences with two fifths of their rows kept: the row operand is gathered by warps of its own, whose waits for a
    free ring slot (16 rounds through rings of a few slots) are bounded like the others.  Calls before and after agree bit for bit."""
    B, k = 40, 200
    batch = W.tiny(B=B, n_vis=[500] * (B - 1) + [431], text_lens=[5] * B, H=8, keep_k=k, seed=605, centres=30)
    c = A.asap_init(0, max_total_tokens=batch.total + B * 500, max_B=B, max_H=8, max_D=1024, max_keep_rows=B * k)
    try:
        inp = A.make_inputs(batch, DEV)
        p = A.Params(keep_k=k)
        names = ("assign", "best_sim", "out_hidden", "out_pos", "src_row", "out_cu_seqlens")
        good = A.alloc_outputs(inp, k, fill=True)
        A.asap_prune_step(c, inp, p, good)
        torch.cuda.synchronize(); A.asap_check(c)
        args = (good.salience.clone(), good.keep_idx.clone(), good.drop_idx.clone())
        for limit in (0, 0, 1, 0, 0):
            out = A.alloc_outputs(inp, k, fill=True)
            if limit:
                A.asap_debug_wait_limit(c, limit)
            A.asap_merge(c, inp, p, *args, out)
            torch.cuda.synchronize()
            if limit:
                with pytest.raises(A.AsapError) as e:
                    A.asap_check(c)
                assert e.value.status == -6 and "timed out in the similarity kernel" in str(e.value)
            else:
                A.asap_check(c)
                _same(good, out, names)
    finally:
        A.asap_free(c)


def test_attention_kernel_gives_up_and_the_context_recovers(ctx):
    batch = W.tiny(B=2, n_vis=[300, 200], text_lens=[30, 11], H=2, keep_k=40, seed=603, centres=6)
    inp = A.make_inputs(batch, DEV)
    p = A.Params(keep_k=40)
    out = A.alloc_outputs(inp, 40, fill=True)
    A.asap_score(ctx, inp, p, out)
    v = W.draw_values(batch, 77).to(DEV)
    scratch = torch.empty(A.asap_attention_scratch_bytes(batch.total, batch.D), dtype=torch.uint8, device=DEV)
    good = torch.zeros_like(v)
    A.asap_attention(ctx, inp, p, out.mask_log, v, scratch, good)
    torch.cuda.synchronize(); A.asap_check(ctx)

    bad = torch.zeros_like(v)
    A.asap_debug_wait_limit(ctx, 1)
    A.asap_attention(ctx, inp, p, out.mask_log, v, scratch, bad)
    torch.cuda.synchronize()
    with pytest.raises(A.AsapError) as e:
        A.asap_check(ctx)
    assert e.value.status == -6 and "timed out in the attention kernel" in str(e.value)

    again = torch.zeros_like(v)
    A.asap_attention(ctx, inp, p, out.mask_log, v, scratch, again)
    torch.cuda.synchronize(); A.asap_check(ctx)
    assert torch.equal(good, again)


@pytest.mark.parametrize("k", [150, 290], ids=["one_slot_tile", "written_bit_matrix"])
def test_consolidation_gives_up_and_the_context_recovers(ctx, k):
    """The similarity kernel gives up and leaves the matrices that the routing reads unwritten (the scratch is filled with
    ones, no valid bit matrix): the routing leaves with its padding, and so does a call made while the bit is still set."""
    batch = W.tiny(B=2, n_vis=[400, 330], text_lens=[9, 12], H=2, keep_k=k, seed=604, centres=20)
    inp = A.make_inputs(batch, DEV)
    p = A.Params(keep_k=k, sim_threshold=0.8)
    out = A.alloc_outputs(inp, k, fill=True)
    A.asap_prune_step(ctx, inp, A.Params(keep_k=k), out)
    torch.cuda.synchronize(); A.asap_check(ctx)
    lists = (out.mass.clone(), out.salience.clone(), out.keep_idx.clone(), out.drop_idx.clone())

    def call():
        scratch = torch.full((A.asap_consolidate_scratch_bytes(2, k),), 255, dtype=torch.uint8, device=DEV)
        o = A.alloc_outputs(inp, k, fill=True)
        n = torch.full((2,), -7, dtype=torch.int32, device=DEV)
        A.asap_consolidate(ctx, inp, p, *lists, scratch, o, n)
        torch.cuda.synchronize()
        return o, n

    good, n_good = call()
    A.asap_check(ctx)
    A.asap_debug_wait_limit(ctx, 1)
    for _ in range(2):                                # the call that gives up, and one that finds the bit set
        bad, n_bad = call()
        assert torch.all(bad.keep_idx == -1) and torch.all(bad.assign == -1) and torch.all(n_bad == 0)
    with pytest.raises(A.AsapError) as e:
        A.asap_check(ctx)
    assert e.value.status == -6 and "timed out in the similarity kernel" in str(e.value)
    again, n_again = call()
    A.asap_check(ctx)
    assert torch.equal(n_good, n_again) and int(n_good.min()) > 0
    _same(good, again, ("keep_idx", "drop_idx", "assign", "best_sim", "out_hidden", "out_pos", "src_row", "out_cu_seqlens"))
