"""The similarity launch picks one of several kernel forms from the problem size.  The large-batch form
(two row tiles per block, kept slots in groups, Sec. 4.2's assignment) is forced here onto small ragged
inputs, so that its edges are compared with the oracle element by element: a second row tile that is
empty, one that is partly filled, several slot groups with a ragged last group, nothing dropped.  The
small-problem form whose slices of the hidden dimension are a thread-block cluster (2, 4 or 8 blocks adding
their partial products through distributed shared memory) is reached with wider hidden states."""
import os

import numpy as np
import pytest
import torch

from oracle import asap_oracle as O
from paper_2603_14549_b200 import binding as A
from paper_2603_14549_b200 import workloads as W
from tests.helpers import bits
from tests.parity import compare_sample, merged_tolerance

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _context(min_blocks, **capacities):
    old = os.environ.get("ASAP_SIM_PAIR_MIN_BLOCKS")
    os.environ["ASAP_SIM_PAIR_MIN_BLOCKS"] = str(min_blocks)          # read once, when the context is made
    try:
        return A.asap_init(0, **capacities)
    finally:
        if old is None:
            del os.environ["ASAP_SIM_PAIR_MIN_BLOCKS"]
        else:
            os.environ["ASAP_SIM_PAIR_MIN_BLOCKS"] = old


@pytest.fixture(scope="module")
def ctx_pair_form():
    c = _context(1, max_total_tokens=40000, max_B=8, max_H=8, max_D=1024, max_keep_rows=8000)
    yield c
    A.asap_free(c)


@pytest.fixture(scope="module")
def ctx_no_pair_form():
    c = _context(1 << 40, max_total_tokens=40000, max_B=20, max_H=16, max_D=2048, max_keep_rows=8000)
    yield c
    A.asap_free(c)


def _merge_matches_oracle(ctx, n_vis, k, H, seed):
    B = len(n_vis)
    batch = W.tiny(B=B, n_vis=n_vis, text_lens=[5 + 3 * b for b in range(B)], H=H, keep_k=k, seed=seed, centres=9)
    p = A.Params(keep_k=k)
    inp = A.make_inputs(batch, DEV)
    mv = inp.max_vis
    sal = torch.zeros(B, mv)
    keep = torch.zeros(B, k, dtype=torch.int32)
    drop = torch.full((B, max(mv - k, 1)), -1, dtype=torch.int32)[:, :mv - k]
    refs = []
    for b in range(B):
        rows = batch.sample_rows(b)
        ref = O.prune_sample(bits(batch.q[rows]), bits(batch.k[rows]), bits(batch.hidden[rows]),
                             batch.pos_ids[rows].numpy(), int(batch.vis_start[b]), int(batch.vis_len[b]),
                             int(batch.text_start[b]), int(batch.text_len[b]), k)
        nv = int(batch.vis_len[b])
        sal[b, :nv] = torch.from_numpy(ref["salience"]).float()
        keep[b] = torch.from_numpy(ref["keep_idx"])
        drop[b, :nv - k] = torch.from_numpy(ref["drop_idx"])
        refs.append(ref)
    out = A.alloc_outputs(inp, k, fill=True)
    A.asap_merge(ctx, inp, p, sal.to(DEV), keep.to(DEV), drop.to(DEV), out)
    torch.cuda.synchronize()
    A.asap_check(ctx)
    ocu = out.out_cu_seqlens.cpu().numpy()
    for b in range(B):
        ref = refs[b]
        nv, v0 = int(batch.vis_len[b]), int(batch.vis_start[b])
        nd = nv - k
        ag = out.assign[b, :nd].cpu().numpy()
        mism = np.nonzero(ag != ref["assign"])[0]
        assert np.all(ref["margin"][mism] <= 1e-4), (b, mism[:8])     # only near-ties may go to another slot
        if nd:
            sim = out.best_sim[b, :nd].cpu().numpy()
            assert np.all(np.abs(sim - ref["best_sim"]) <= 2e-4), b
        rows = batch.sample_rows(b)
        ref2 = O.prune_sample(bits(batch.q[rows]), bits(batch.k[rows]), bits(batch.hidden[rows]),
                              batch.pos_ids[rows].numpy(), v0, nv, int(batch.text_start[b]),
                              int(batch.text_len[b]), k, assign_override=ag)
        gh = O.bf16_bits_to_f64(bits(out.out_hidden[int(ocu[b]):int(ocu[b + 1])].cpu()))
        assert np.all(np.abs(gh - ref2["out_hidden"]) <= merged_tolerance(ref2["out_hidden"])), b
        assert np.array_equal(out.out_pos[int(ocu[b]):int(ocu[b + 1])].cpu().numpy(), ref2["out_pos"])


@pytest.fixture(scope="module")
def ctx_default():
    c = A.asap_init(0, max_total_tokens=40000, max_B=8, max_H=8, max_D=1024, max_keep_rows=8000)
    yield c
    A.asap_free(c)


@pytest.mark.parametrize("n_vis,k,H", [
    ([300, 129], 100, 8),        # hidden size 1024: eight slices per row tile, ragged last row tiles
    ([640], 256, 8),             # the widest single slot tile, 384 dropped rows
    ([200, 130, 131], 16, 4),    # hidden size 512: four slices, one narrow slot tile
    ([129, 129, 129, 129, 129, 129, 129, 129], 33, 8),   # sixteen row tiles: fewer slices per tile
])
def test_cluster_form_matches_the_oracle(ctx_default, n_vis, k, H):
    _merge_matches_oracle(ctx_default, n_vis, k, H, seed=933)


@pytest.mark.parametrize("n_vis,k", [
    ([520, 300, 257], 40),      # three / two / two row tiles: pairs with a full, a partial and an empty second tile
    ([600, 513], 257),          # two groups of 144 slots, the second ragged (113 slots)
    ([256, 300], 256),          # sample 0 drops nothing
    ([129, 1000], 17),          # one group narrower than an MMA's smallest useful width
])
def test_pair_form_matches_the_oracle(ctx_pair_form, n_vis, k):
    _merge_matches_oracle(ctx_pair_form, n_vis, k, H=2, seed=911)


@pytest.mark.parametrize("n_vis,k,H", [
    ([700, 650], 257, 2),        # two accumulators in one pass, the second ragged
    ([700, 650], 384, 2),        # ... and full
    ([700, 650], 512, 2),        # two accumulators in turn, two passes
    ([700, 650], 600, 2),        # three
    ([700], 300, 16),            # slices of the hidden dimension that add up through global memory
    ([900], 600, 16),
    ([1300] * 19 + [1041], 260, 2),   # more row tiles than SMs: not sliced, and too few slots kept to be gathered
], ids=["wide_ragged", "wide_full", "two_passes", "three_passes", "sliced_wide", "sliced", "large"])
def test_several_slot_tiles_without_the_pair_form(ctx_no_pair_form, n_vis, k, H):
    """More than 256 kept slots take two row tiles per block, unless that form's partial results outgrow their buffer (above a
    million visual rows): the forms that serve such a batch, on small ones."""
    _merge_matches_oracle(ctx_no_pair_form, n_vis, k, H, seed=935)


@pytest.mark.parametrize("nv,k,H", [(700, 300, 2), (1300, 600, 2), (700, 300, 16), (500, 150, 16)],
                         ids=["two_tiles", "three_tiles", "sliced", "cluster"])
def test_kept_rows_matrix_without_the_pair_form(ctx_no_pair_form, nv, k, H):
    """The same for the matrix of the kept rows' similarities; the routing then forms its bit matrix itself."""
    from tests.test_gpu_consolidate import _check, _run
    batch = W.tiny(B=2, n_vis=[nv, nv - 40], text_lens=[4, 9], H=H, keep_k=k, seed=936, centres=k // 8)
    out, n_abs, st1 = _run(ctx_no_pair_form, batch, k, 0.8, stage1=lambda bt, b, kk: W.random_stage1(bt, b, kk, 33))
    assert _check(batch, k, 0.8, out, n_abs, st1) > 0


def test_many_kept_slots_of_a_long_sequence():
    """A third of 15000 rows kept: enough for the gathered form, but the grouping's counters do not fit its shared memory; the
    tiled form with its fewer warps takes the call (20 slot tiles that share two accumulators)."""
    c = A.asap_init(0, max_total_tokens=31000, max_B=2, max_H=2, max_D=256, max_keep_rows=10000)
    try:
        _merge_matches_oracle(c, [15000, 5100], 5000, H=2, seed=934)
    finally:
        A.asap_free(c)


def test_pair_form_at_the_end_of_its_partial_results():
    """2990 pairs of row tiles with four groups of slots each: close to the most that the form takes, and more than its partial results
    had room for before the groups left a share of the row norms each.  115 copies of two sequences give the same bits, and the first
    two are the oracle's."""
    two = W.tiny(B=2, n_vis=[3100, 3081], text_lens=[8, 5], H=1, keep_k=770, seed=937, centres=60)
    n, reps = two.total, 115
    rep = lambda t: t.repeat(reps, *([1] * (t.dim() - 1)))
    cu = torch.cat([torch.zeros(1, dtype=torch.int32)] + [two.cu_seqlens[1:] + r * n for r in range(reps)]).to(torch.int32)
    batch = W.Batch(name="tiny", B=2 * reps, H=1, head_dim=128, D=128, keep_k=770, cu_seqlens=cu,
                    **{f: rep(getattr(two, f)) for f in ("vis_start", "vis_len", "text_start", "text_len", "q", "k", "hidden", "pos_ids")})
    p = A.Params(keep_k=770)
    c = A.asap_init(0, max_total_tokens=batch.total + batch.B * 20, max_B=batch.B, max_H=1, max_D=128, max_keep_rows=batch.B * 770)
    try:
        inp = A.make_inputs(batch, DEV)
        out = A.alloc_outputs(inp, 770, fill=True)
        A.asap_prune_step(c, inp, p, out)
        torch.cuda.synchronize()
        A.asap_check(c)
    finally:
        A.asap_free(c)
    for b in range(2):
        compare_sample(batch, b, p, out)
    for f in ("rank_score", "keep_idx", "assign", "best_sim"):
        t = getattr(out, f)
        assert torch.equal(t.view(reps, -1), t[:2].reshape(1, -1).expand(reps, -1)), f
    rows = int(out.out_cu_seqlens[2])
    h = out.out_hidden[:reps * rows].view(reps, -1)
    assert torch.equal(h, h[:1].expand(reps, -1))


def test_pair_form_gives_up_and_the_context_recovers(ctx_pair_form):
    """The bounded waits of this form, in the harmless way: the wait limit of one call is a single clock
    cycle, the call returns, the status names the kernel, and the next call is a fresh one bit for bit."""
    ctx = ctx_pair_form
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
    for n in ("assign", "best_sim", "out_hidden", "out_pos", "src_row", "out_cu_seqlens"):
        assert torch.equal(getattr(ref, n), getattr(again, n)), n
