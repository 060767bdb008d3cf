"""What a program that prunes visual tokens asks of this library, with the sizes it asks for.

Four kinds of pass, each through the public entry points of ``paper_2603_14549_b200.binding``:

  step         asap_prune_step once, or several times in succession (a progressive schedule), on a packed batch
  attention    asap_attention: the layer's attention under the mask of Eq. 3, every row of the batch
  consolidate  asap_consolidate: stage 2 in the wording of Sec. 4.2, on stage 1's lists
  kv           asap_compact_kv: the cached keys and values of the layers before the prune step

Inputs are drawn on the GPU from the seed alone.  Queries and keys are N(0, 1) entries (a rotary embedding
leaves that distribution as it is) plus one shared direction per head along which the visual keys carry a relevance:
keep_k tokens of a sequence are relevant, the others are background, and the two groups are apart by
more than the spread that the random part causes.  (Rankings without such a gap are decided by the last bit of a
sum, and two correct implementations then keep different tokens.)  Visual hidden rows are a cluster centre plus a variation in a
few directions plus noise, so that the most similar kept token stands out for all but a few rows in a million.
"""
from __future__ import annotations

import math
import random
import weakref

import torch

from paper_2603_14549_b200 import binding as A

DEVICE = "cuda:0"
SYSTEM = 35            # rows of the system prompt in front of the image span
HEAD_DIM = 128
VARIATION_RANK = 24    # directions in which the rows of one cluster differ


def _step(**kw):
    c = {"what": "step", "B": 1, "vis_lo": 576, "vis_hi": 576, "text_lo": 32, "text_hi": 32, "H": 32, "keep": 192,
         "steps": 1, "shape": 1, "centres": 64, "outliers": 0.0, "lambda_max": 1.0, "threshold": -1.0,
         "per_head": False, "visual_rows": 0}
    c.update(kw)
    return c


def listed():
    return [
        # one request with one image: latency
        _step(name="step_one_image"),
        # a batch of short chats, one image each, a tight budget
        _step(name="step_chat_batch", B=16, text_lo=16, text_hi=128, keep=64, shape=2),
        # images of four tiles, some rows with ten times the norm (attention sinks)
        _step(name="step_tiles", B=8, vis_lo=2304, vis_hi=2304, text_lo=64, text_hi=64, keep=320, centres=192, outliers=0.02),
        # the largest batch that one GPU is given: full-resolution images, long and short questions
        _step(name="step_anyres_large", B=64, vis_lo=2880, vis_hi=2880, text_lo=32, text_hi=256, keep=576, shape=3),
        # the wider model, pruned at three layers: 2304 -> 1152 -> 576 -> 288 tokens, each step on the last one's result
        _step(name="step_schedule_wide", B=32, vis_lo=2304, vis_hi=2304, text_lo=128, text_hi=128, H=40, keep=1152, steps=3,
              centres=192),
        # images of every size in one batch, odd lengths, a threshold on the similarity, half the leak
        _step(name="step_mixed_images", B=12, vis_lo=577, vis_hi=2881, text_lo=17, text_hi=201, keep=145, shape=4,
              lambda_max=0.5, threshold=0.5),
        # a mask per head, the last visual rows among the ranking rows
        _step(name="step_per_head_rows", B=8, vis_lo=1536, vis_hi=1536, text_lo=64, text_hi=64, keep=340, per_head=True,
              visual_rows=32, lambda_max=0.5),
        # stage 2 inside the kept set, for a caller that has ranked the tokens
        {"name": "consolidate_anyres", "what": "consolidate", "B": 24, "vis_lo": 2880, "vis_hi": 2880, "text_lo": 32,
         "text_hi": 256, "H": 32, "keep": 576, "shape": 5, "centres": 64, "threshold": 0.8},
        # the masked attention of one request, of a batch of chats and of the largest batch
        {"name": "attention_one_image", "what": "attention", "B": 1, "vis_lo": 576, "vis_hi": 576, "text_lo": 32, "text_hi": 32,
         "H": 32, "shape": 1, "mask": True},
        {"name": "attention_chat_batch", "what": "attention", "B": 16, "vis_lo": 576, "vis_hi": 576, "text_lo": 16,
         "text_hi": 128, "H": 32, "shape": 2, "mask": True},
        {"name": "attention_anyres_large", "what": "attention", "B": 64, "vis_lo": 2880, "vis_hi": 2880, "text_lo": 32,
         "text_hi": 256, "H": 32, "shape": 3, "mask": True},
        # keys and values of three layers after the step of the chat batch
        {"name": "kv_chat_batch", "what": "kv", "B": 16, "vis_lo": 576, "vis_hi": 576, "text_lo": 16, "text_hi": 128, "H": 32,
         "keep": 64, "shape": 2, "tensors": 6},
    ]


MOST_ELEMENTS = 64 * (SYSTEM + 2880 + 144) * 4096      # packed rows x width of the largest listed batch


def draw(rng):
    """A case of the same ranges: batches of 1 to 64, images of 144 to 2881 tokens, questions of 8 to 256."""
    log_int = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    what = rng.choice(["step", "step", "step", "step", "attention", "attention", "consolidate", "kv"])
    H = rng.choice([16, 20, 32, 32, 40])
    vis_hi = log_int(144, 2881)
    vis_lo = vis_hi if rng.random() < 0.5 else log_int(max(144, vis_hi // 3), vis_hi)
    text_lo = log_int(8, 128)
    text_hi = rng.randint(text_lo, 256)
    B = log_int(1, 64)
    B = max(1, min(B, MOST_ELEMENTS // ((SYSTEM + vis_hi + text_hi) * H * HEAD_DIM)))
    c = {"what": what, "B": B, "vis_lo": vis_lo, "vis_hi": vis_hi, "text_lo": text_lo, "text_hi": text_hi, "H": H,
         "shape": rng.randint(1, 1 << 20)}
    if what == "attention":
        c["mask"] = rng.random() < 0.8
        return c
    c["keep"] = min(vis_lo, max(16, log_int(max(1, vis_lo // 10), max(2, vis_lo // 2))))
    if what == "kv":
        c["tensors"] = 2 * rng.randint(1, 4)
        return c
    if what == "consolidate":
        c["keep"] = min(c["keep"], vis_lo - 1)
        c.update(centres=max(2, c["keep"] // rng.randint(2, 9)), threshold=0.8)
        return c
    option = rng.choice(["plain", "plain", "threshold", "rows", "per_head"])
    return _step(**c, centres=rng.choice([32, 64, 192]), outliers=rng.choice([0.0, 0.0, 0.02]),
                 threshold=0.5 if option == "threshold" else -1.0, lambda_max=rng.choice([1.0, 1.0, 0.5]),
                 per_head=option == "per_head", visual_rows=max(1, min(32, text_lo // 2)) if option in ("rows", "per_head") else 0)


# ------------------------------------------------------------------------------------------- shapes
def _lengths(case):
    r = random.Random(case["shape"])
    vis = [r.randint(case["vis_lo"], case["vis_hi"]) for _ in range(case["B"])]
    text = [r.randint(case["text_lo"], case["text_hi"]) for _ in range(case["B"])]
    vis[0], text[0] = case["vis_hi"], case["text_hi"]
    return vis, text


def _keeps(case):
    return [case["keep"] >> i for i in range(case.get("steps", 1))]


class Handle:
    """A library context, given back when the program drops it."""

    def __init__(self, tokens, B, H, keep_rows):
        self.ctx = A.asap_init(0, tokens, B, H, H * HEAD_DIM, keep_rows)
        weakref.finalize(self, A.asap_free, self.ctx)


def _inputs(vis, text, H, q, k, hidden, pos, rank=None):
    seq = [SYSTEM + v + t for v, t in zip(vis, text)]
    cu = [0]
    for n in seq:
        cu.append(cu[-1] + n)
    dev = lambda v: torch.tensor(v, dtype=torch.int32, device=DEVICE)
    text_start = [SYSTEM + v for v in vis]
    rank_start = [s - rank for s in text_start] if rank else None
    rank_len = [t + rank for t in text] if rank else None
    return A.Inputs(B=len(vis), H=H, head_dim=HEAD_DIM, D=H * HEAD_DIM, total_tokens=cu[-1], min_vis=min(vis), max_vis=max(vis),
                    max_seq=max(seq), max_rank=max(rank_len or text), cu_seqlens=dev(cu), vis_start=dev([SYSTEM] * len(vis)),
                    vis_len=dev(vis), text_start=dev(text_start), text_len=dev(text), q=q, k=k, hidden=hidden, pos_ids=pos,
                    rank_start=dev(rank_start) if rank else None, rank_len=dev(rank_len) if rank else None)


# ------------------------------------------------------------------------------------------- values
def _normal(gen, *shape):
    return torch.randn(*shape, generator=gen, device=DEVICE, dtype=torch.bfloat16)


def _queries_keys(gen, vis, text, H, keep):
    """q, k [tokens, H, 128]; `keep` relevant visual keys per sequence (None: no relevance)."""
    total = sum(SYSTEM + v + t for v, t in zip(vis, text))
    q, k = _normal(gen, total, H, HEAD_DIM), _normal(gen, total, H, HEAD_DIM)
    row = 0
    for v, t in zip(vis, text):
        n = SYSTEM + v + t
        if keep is not None:
            u = _normal(gen, H, HEAD_DIM)
            rel = torch.rand(v, generator=gen, device=DEVICE) * 1.5 - 1.5
            who = torch.randperm(v, generator=gen, device=DEVICE)[:keep]
            rel[who] = torch.rand(keep, generator=gen, device=DEVICE) + 1.5
            q[row:row + n] += 0.5 * u
            k[row + SYSTEM:row + SYSTEM + v] += (rel * (2.0 / math.sqrt(HEAD_DIM))).to(torch.bfloat16)[:, None, None] * u
        row += n
    return q, k


def _hidden(gen, vis, text, D, centres, variation, outliers):
    total = sum(SYSTEM + v + t for v, t in zip(vis, text))
    hidden = _normal(gen, total, D)
    basis = _normal(gen, VARIATION_RANK, D)
    row = 0
    for v, t in zip(vis, text):
        rows = hidden[row + SYSTEM:row + SYSTEM + v]
        rows *= 0.3
        rows += _normal(gen, centres, D)[torch.randint(0, centres, (v,), generator=gen, device=DEVICE)]
        if variation:
            rows += (_normal(gen, v, VARIATION_RANK) * (variation / math.sqrt(VARIATION_RANK))) @ basis
        if outliers:
            rows[torch.randperm(v, generator=gen, device=DEVICE)[:max(1, int(round(outliers * v)))]] *= 10.0
        row += SYSTEM + v + t
    return hidden


def _positions(vis, text):
    return torch.cat([torch.arange(SYSTEM + v + t, dtype=torch.int32, device=DEVICE) for v, t in zip(vis, text)])


def prepare(case, seed):
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)
    vis, text = _lengths(case)
    B, H = case["B"], case["H"]
    D = H * HEAD_DIM
    total = sum(SYSTEM + v + t for v, t in zip(vis, text))
    tokens = max(total, B * max(vis))
    what = case["what"]

    if what == "step":
        params, inputs, outputs = [], [], []
        hidden = _hidden(gen, vis, text, D, case["centres"], 0.6, case["outliers"])
        pos = _positions(vis, text)
        for keep in _keeps(case):
            q, k = _queries_keys(gen, vis, text, H, keep)
            inputs.append(_inputs(vis, text, H, q, k, hidden, pos, case["visual_rows"]))
            params.append(A.Params(keep_k=keep, lambda_max=case["lambda_max"], per_head_mask=case["per_head"],
                                   sim_threshold=case["threshold"] if case["threshold"] > -1.0 else -math.inf))
            outputs.append(A.alloc_outputs(inputs[-1], keep, fill=True, per_head=case["per_head"]))
            hidden, pos, vis = outputs[-1].out_hidden, outputs[-1].out_pos, [keep] * B     # the next step's
        return {"what": what, "handle": Handle(tokens, B, H, B * case["keep"]), "inputs": inputs, "params": params, "outputs": outputs}

    if what == "attention":
        q, k = _queries_keys(gen, vis, text, H, None)
        v = _normal(gen, total, H, HEAD_DIM)
        mask = torch.log(torch.clamp(torch.rand(B, max(vis), generator=gen, device=DEVICE), min=1e-6)) if case["mask"] else None
        scratch = torch.empty(A.asap_attention_scratch_bytes(total, D), dtype=torch.uint8, device=DEVICE)
        return {"what": what, "handle": Handle(tokens, B, H, B), "inputs": _inputs(vis, text, H, q, k, None, None),
                "params": A.Params(keep_k=1, mask_enable=case["mask"]), "mask": mask, "v": v, "scratch": scratch,
                "out": torch.zeros_like(v)}

    keep = case["keep"]
    perms = [torch.randperm(v, generator=gen, device=DEVICE).to(torch.int32) for v in vis]
    kept = torch.stack([torch.sort(p[:keep]).values for p in perms])

    if what == "consolidate":
        hidden = _hidden(gen, vis, text, D, case["centres"], 0.0, 0.0)
        inp = _inputs(vis, text, H, None, None, hidden, _positions(vis, text))
        drop = torch.full((B, max(vis) - keep), -1, dtype=torch.int32, device=DEVICE)
        for b, p in enumerate(perms):
            drop[b, :vis[b] - keep] = torch.sort(p[keep:]).values
        mass = torch.exp(torch.randn(B, max(vis), generator=gen, device=DEVICE))
        salience = torch.rand(B, max(vis), generator=gen, device=DEVICE)
        return {"what": what, "handle": Handle(tokens, B, H, B * keep), "inputs": inp, "mass": mass, "salience": salience,
                "kept": kept, "drop": drop, "params": A.Params(keep_k=keep, sim_threshold=case["threshold"]),
                "scratch": torch.empty(A.asap_consolidate_scratch_bytes(B, keep), dtype=torch.uint8, device=DEVICE),
                "outputs": A.alloc_outputs(inp, keep, fill=True), "absorbed": torch.zeros(B, dtype=torch.int32, device=DEVICE)}

    rows, row = [], 0
    for b, (v, t) in enumerate(zip(vis, text)):
        rows += [torch.arange(row, row + SYSTEM, dtype=torch.int32, device=DEVICE), kept[b] + (row + SYSTEM),
                 torch.arange(row + SYSTEM + v, row + SYSTEM + v + t, dtype=torch.int32, device=DEVICE)]
        row += SYSTEM + v + t
    src_row = torch.cat(rows)
    src = [_normal(gen, total, D) for _ in range(case["tensors"])]
    return {"what": what, "handle": Handle(tokens, B, H, B * keep), "src_row": src_row, "src": src,
            "n_rows": torch.tensor([src_row.numel()], dtype=torch.int32, device=DEVICE),
            "dst": [torch.zeros(src_row.numel(), D, dtype=torch.bfloat16, device=DEVICE) for _ in src]}


# ------------------------------------------------------------------------------------------- one pass
def _fields(out, names):
    return {n: getattr(out, n) for n in names if getattr(out, n) is not None}


LISTS = ["keep_idx", "drop_idx", "assign", "best_sim", "out_hidden", "out_pos", "src_row", "out_cu_seqlens"]


def run(state):
    ctx, what = state["handle"].ctx, state["what"]
    if what == "step":
        for inp, params, out in zip(state["inputs"], state["params"], state["outputs"]):
            A.asap_prune_step(ctx, inp, params, out)
        return [_fields(out, ["mass", "salience", "mask_log", "mask_log_heads", "rank_score"] + LISTS) for out in state["outputs"]]
    if what == "attention":
        A.asap_attention(ctx, state["inputs"], state["params"], state["mask"], state["v"], state["scratch"], state["out"])
        return state["out"]
    if what == "consolidate":
        A.asap_consolidate(ctx, state["inputs"], state["params"], state["mass"], state["salience"], state["kept"], state["drop"],
                           state["scratch"], state["outputs"], state["absorbed"])
        return _fields(state["outputs"], LISTS), state["absorbed"]
    A.asap_compact_kv(ctx, state["src_row"], state["n_rows"], state["src"], state["dst"])
    return state["dst"]


# ------------------------------------------------------------------------------------------- bounds
def work(case):
    """Every input row that matters read once, every output row written once; multiply-adds of the contractions."""
    vis, text = _lengths(case)
    D = case["H"] * HEAD_DIM
    row = 2 * D
    nbytes = flops = 0
    for v, t in zip(vis, text):
        n = SYSTEM + v + t
        if case["what"] == "attention":
            nbytes += 4 * n * row
            flops += 4 * D * (n * (n + 1) // 2 + (v * (v - 1) // 2 if case["mask"] else 0))
        elif case["what"] == "kv":
            nbytes += 2 * (n - v + case["keep"]) * row * case["tensors"]
        elif case["what"] == "consolidate":
            k = case["keep"]
            nbytes += (n + n - v + k) * row
            flops += k * (k - 1) * D + 2 * v * D
        else:
            for k in _keeps(case):
                n, r = SYSTEM + v + t, t + case["visual_rows"]
                nbytes += (v + t) * row + n * row + (n + n - v + k) * row + 4 * (4 * v + 2 * v)
                flops += 3 * v * D + 2 * r * (n - r // 2) * D + 2 * (v - k) * k * D + 2 * v * D
                v = k
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """bf16 results of fp32 sums.  Against float64 the one rounding of a merged row is a relative error of 1.7e-3,
    and the attention, whose probabilities are rounded too, shows 2.0e-3 and at most 2.4e-2 of the root mean square.
    Two orders of summation give the same kept sets and assignments on all cases, and a largest difference of one bf16
    step (9e-3); should a row be sent to another of two equally similar kept tokens, two merged rows change by more."""
    if case["what"] == "kv":
        return "exact"
    if case["what"] == "attention":
        return {"rel": 8e-3, "max": 0.1}
    return {"rel": 7e-3, "max": 0.3, "differ": 5e-4}
