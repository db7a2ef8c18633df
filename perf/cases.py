"""What a program that runs SparseD's denoising loop asks of this library, as timed cases.

One pass of a case is one attention call of one denoising step, made through the Python binding the way a model's
attention layer makes it. ``phase`` says which step of the schedule it is:

* ``full``    a step before the switch step: dense attention (``sparsed_attention_step``)
* ``switch``  the switch step: dense attention, then the pattern is selected from that very pass
* ``sparse``  a step after it: block-sparse attention on the pattern in hand
* ``select``  a pattern selected from Q and K alone, or with the LSE of an earlier dense pass
              (``sparsed_select_pattern``: what a step without pattern reuse, or a caller with its own dense kernel, runs)

Sizes are those of the repository's workloads (``synthetic.CONFIGS``, the block-32 short-context setting of the
benchmark) and generic ones between them. Inputs are its synthetic layers: N(0,1)/sqrt(d) queries and keys with planted
bands, sinks and stripes, at ``norm`` 3 (attention close to uniform) up to 12 (sharp heads, logit boost 12.7).
``layout`` is how the tensors lie in memory: ``head`` = [B, H, L, D], ``token`` = a transposed view of [B, L, H, D], as a
projection's output is.
"""
from __future__ import annotations

import math

import torch

import paper_2509_24014_b200 as sd
from paper_2509_24014_b200 import synthetic

HEAD_DIM = 128
TOTAL_STEPS, SKIP = 64, 0.2
STEP_OF = {"full": 1, "switch": 12, "sparse": 13}   # 1-based; floor(64 * 0.2) = 12 is the switch step

# Bounds of a drawn case: what the largest listed one needs.
MOST_LOGITS = 32 * 65536 * 65536           # batch * query heads * tokens^2
MOST_ELEMENTS = 32 * 65536 * HEAD_DIM      # of Q
MOST_STATS = 32 * 65536 * 65536 // 128     # row statistics of the switch step


def _case(name, phase, batch, heads_q, heads_kv, tokens, block, keep, prompt, norm, layout, lse=False,
          scores=False):
    return {"name": name, "phase": phase, "batch": batch, "heads_q": heads_q, "heads_kv": heads_kv, "tokens": tokens,
            "block": block, "keep": keep, "prompt": prompt, "norm": norm, "layout": layout, "lse": lse,
            "scores": scores}


def listed():
    return [
        # A layer (or a tensor-parallel slice of one) of two heads over 1024 tokens: the smallest calls, where
        # launches, host work and the length of one thread block's chain are what is paid for.
        _case("two_heads_1k_full", "full", 1, 2, 2, 1024, 64, 0.3, 0, 3.0, "head"),
        _case("two_heads_1k_sparse_b64", "sparse", 1, 2, 2, 1024, 64, 0.3, 0, 3.0, "head"),
        # A short conversation whose length is not a multiple of anything: dense attention takes any length.
        _case("ragged_1900_full", "full", 1, 32, 32, 1900, 64, 0.3, 0, 6.0, "token"),
        # The short-context setting (32-key blocks, half of them kept), one request at its switch step ...
        _case("short_4k_switch_b32", "switch", 1, 32, 32, 4096, 32, 0.5, 2048, 6.0, "token"),
        # ... and a batch of eight in the sparse phase, where a denoising loop spends most of its steps.
        _case("short_4k_batch8_sparse_b32", "sparse", 8, 32, 32, 4096, 32, 0.5, 2048, 3.0, "head"),
        # An 8k LLaDA-shaped layer (half prompt, half generation) through the three phases of the loop.
        _case("llada_8k_full", "full", 1, 32, 32, 8192, 128, 0.2, 4096, 3.0, "head"),
        _case("llada_8k_switch", "switch", 1, 32, 32, 8192, 128, 0.2, 4096, 12.0, "head"),
        _case("llada_8k_sparse", "sparse", 1, 32, 32, 8192, 128, 0.2, 4096, 3.0, "head"),
        # A 16k Dream-shaped layer with grouped heads: its sparse phase, and a step that selects afresh from its Q and K
        # (with the block scores beside the lists, as a program that studies its patterns takes them).
        _case("dream_16k_sparse", "sparse", 1, 28, 4, 16384, 128, 0.15, 0, 12.0, "token"),
        _case("dream_16k_select", "select", 1, 28, 4, 16384, 128, 0.15, 0, 3.0, "token", scores=True),
        # The 64k loop: the sparse phase, which is four fifths of its steps, and the heaviest single call.
        _case("loop_64k_sparse", "sparse", 1, 32, 32, 65536, 128, 0.1, 0, 3.0, "head"),
        _case("loop_64k_switch", "switch", 1, 32, 32, 65536, 128, 0.1, 0, 3.0, "head"),
    ]


def draw(rng):
    while True:
        # by how often a loop makes the call
        phase = rng.choice(["full", "full", "switch", "sparse", "sparse", "sparse", "select"])
        heads_q, heads_kv = rng.choice([(2, 2), (8, 8), (16, 4), (28, 4), (32, 8), (32, 32)])
        tokens = int(math.exp(rng.uniform(math.log(512), math.log(65536))))
        if tokens <= 2048:
            block = rng.choice([32, 64])
        elif tokens <= 8192:
            block = rng.choice([32, 64, 128])
        else:
            block = rng.choice([64, 128, 128, 128])
        if phase != "full":
            tokens -= tokens % block
        batch = rng.choice([1, 1, 1, 2, 3, 8]) if tokens <= 8192 else 1
        keep = round(rng.uniform(0.3, 0.5) if block == 32 else rng.uniform(0.08, 0.3), 3)
        prompt = 0 if rng.random() < 0.4 else int(tokens * rng.uniform(0.2, 0.8)) // block * block
        rows = batch * heads_q * tokens
        if rows * tokens > MOST_LOGITS or rows * HEAD_DIM > MOST_ELEMENTS or rows * tokens // block > MOST_STATS:
            continue
        c = _case("", phase, batch, heads_q, heads_kv, tokens, block, keep, prompt, rng.choice([3.0, 6.0, 9.0, 12.0]),
                  rng.choice(["head", "token"]), phase == "select" and rng.random() < 0.5,
                  phase == "select" and rng.random() < 0.5)
        del c["name"]
        return c


def _params(case):
    return sd.make_params(case["block"], case["keep"], case["prompt"])


def _inputs(case, seed):
    cfg = synthetic.AttnConfig("perf", case["batch"], case["heads_q"], case["heads_kv"], case["tokens"], HEAD_DIM,
                               case["block"], case["keep"], case["prompt"], seed=seed, plant_norm=case["norm"])
    q, k, v = synthetic.make_qkv(cfg, torch.device("cuda"))
    if case["layout"] == "token":
        q, k, v = (t.transpose(1, 2).contiguous().transpose(1, 2) for t in (q, k, v))
    return q, k, v


def _mean_scores(q, k, block):
    """Block-mean scores, taken with plain tensor operations. A loop's pattern is ranked on these here (on these inputs
    they keep 98-99 % of the blocks the exact scores do), so that it is the same pattern whatever the scoring kernels'
    rounding is."""
    B, H, L, D = q.shape
    bs, nb, group = block, L // block, H // k.shape[1]
    scores = torch.empty(B, H, nb, nb, dtype=torch.float32, device=q.device)
    for b in range(B):
        for h in range(H):
            mq = q[b, h].float().reshape(nb, bs, D).mean(1)
            mk = k[b, h // group].float().reshape(nb, bs, D).mean(1)
            scores[b, h] = torch.softmax(mq @ mk.t() / math.sqrt(D), dim=-1)
    return scores


def _pattern_from_means(q, k, case, params, ws):
    """The pattern a loop in its sparse phase has in hand."""
    B, H, L, _ = q.shape
    nb, scores = L // case["block"], _mean_scores(q, k, case["block"])
    k_pre, k_gen = sd.sparsed_kept_per_row(params, L)
    pat, row_ptr, col_idx = sd.new_pattern(B, H, nb, k_pre + k_gen, q.device)
    sd.sparsed_select_from_scores(scores, params, pat, ws)
    return pat, row_ptr, col_idx


def prepare(case, seed):
    q, k, v = _inputs(case, seed)
    dev = q.device
    state = {"phase": case["phase"], "q": q, "k": k, "v": v, "params": _params(case), "lse": None, "scores": None}
    params, phase = state["params"], case["phase"]
    if phase == "select":
        nbytes = sd.sparsed_workspace_bytes(sd.OP_SELECT_PATTERN, sd.make_shape(q, k), params)
    elif phase == "switch":
        nbytes = sd.sparsed_workspace_bytes(sd.OP_ATTENTION_STEP, sd.make_shape(q, k), params)
    else:
        nbytes = sd.sparsed_workspace_bytes(sd.OP_ATTN_FULL)
    state["ws"] = sd.new_workspace(nbytes, dev)
    if phase != "select":
        state["o"] = torch.empty_like(q)
    if phase == "full":
        # the loop's pattern buffers exist from its first step on; nothing reads or writes them yet
        state["pattern"] = sd.Pattern()
    elif phase == "sparse":
        state["pattern"], state["row_ptr"], state["col_idx"] = _pattern_from_means(q, k, case, params, state["ws"])
    else:
        k_pre, k_gen = sd.sparsed_kept_per_row(params, case["tokens"])
        state["pattern"], state["row_ptr"], state["col_idx"] = sd.new_pattern(
            case["batch"], case["heads_q"], case["tokens"] // case["block"], k_pre + k_gen, dev)
    if case["scores"]:
        nb = case["tokens"] // case["block"]
        state["scores"] = torch.empty(case["batch"], case["heads_q"], nb, nb, dtype=torch.float32, device=dev)
    if case["lse"]:
        lse = torch.empty(q.shape[:3], dtype=torch.float32, device=dev)
        sd.sparsed_attn_full(q, k, v, torch.empty_like(q), lse, state["ws"])
        state["lse"] = lse
    return state


def run(state):
    phase = state["phase"]
    if phase == "select":
        sd.sparsed_select_pattern(state["q"], state["k"], state["params"], state["pattern"], state["ws"],
                                  lse=state["lse"], scores_out=state["scores"])
        out = {"row_ptr": state["row_ptr"], "col_idx": state["col_idx"]}
        if state["scores"] is not None:
            out["scores"] = state["scores"]
        return out
    sd.sparsed_attention_step(state["q"], state["k"], state["v"], state["o"], state["params"], STEP_OF[phase],
                              TOTAL_STEPS, SKIP, state["pattern"], state["ws"])
    if phase == "switch":
        return {"o": state["o"], "row_ptr": state["row_ptr"], "col_idx": state["col_idx"]}
    return {"o": state["o"]}


def _kept_blocks(scores, case):
    """[nb, kept] ids of the blocks that each row of a head's scores keeps: the best of the prompt's blocks and of the
    others, each ranked by itself, ties to the lower id, in ascending order."""
    nb, ids, first = scores.shape[-1], [], 0
    split = case["prompt"] // case["block"]
    for end in ([split] if 0 < split < nb else []) + [nb]:
        kept = min(max(math.ceil(case["keep"] * (end - first) - 1e-6), 1), end - first)
        order = torch.sort(scores[:, first:end], dim=-1, descending=True, stable=True).indices[:, :kept]
        ids.append(order + first)
        first = end
    return torch.cat(ids, dim=-1).sort(dim=-1).values


def exact(case, seed):
    """What run() returns, from plain tensor operations in 64 bits. Lists of blocks that are chosen by exact scores have no
    such value here: see tolerance()."""
    if case["phase"] == "select" and not case["scores"]:
        return None
    q, k, v = _inputs(case, seed)
    B, H, L, D = q.shape
    bs, nb, group = case["block"], L // case["block"], H // k.shape[1]
    o = torch.empty(B, H, L, D, dtype=torch.float64, device=q.device) if case["phase"] != "select" else None
    pooled = torch.empty(B, H, nb, nb, dtype=torch.float64, device=q.device) if case["phase"] == "select" else None
    means = _mean_scores(q, k, bs) if case["phase"] == "sparse" else None
    for b in range(B):
        for h in range(H):
            qh = q[b, h].double() / math.sqrt(D)
            kh, vh = k[b, h // group].double(), v[b, h // group].double()
            if case["phase"] == "sparse":
                ids = _kept_blocks(means[b, h], case)
                step = max(1, (1 << 25) // (ids.shape[1] * bs * D))
                kb, vb, qb = kh.reshape(nb, bs, D), vh.reshape(nb, bs, D), qh.reshape(nb, bs, D)
                for i in range(0, nb, step):
                    at = ids[i:i + step]
                    p = torch.softmax(qb[i:i + step] @ kb[at].flatten(1, 2).transpose(1, 2), dim=-1)
                    o[b, h, i * bs:(i + step) * bs] = (p @ vb[at].flatten(1, 2)).flatten(0, 1)
                continue
            step = max(bs, (1 << 27) // L // bs * bs)
            for i in range(0, L, step):
                p = torch.softmax(qh[i:i + step] @ kh.t(), dim=-1)
                if pooled is not None:
                    pooled[b, h, i // bs:(i + step) // bs] = p.reshape(-1, bs, nb, bs).mean(dim=(1, 3))
                else:
                    o[b, h, i:i + step] = p @ vh
    if case["phase"] == "select":
        return {"row_ptr": None, "col_idx": None, "scores": pooled}
    if case["phase"] == "switch":
        return {"o": o, "row_ptr": None, "col_idx": None}
    return {"o": o}


def work(case):
    B, Hq, Hkv, L = case["batch"], case["heads_q"], case["heads_kv"], case["tokens"]
    q_bytes, kv_bytes = 2 * B * Hq * L * HEAD_DIM, 2 * B * Hkv * L * HEAD_DIM
    logits = B * Hq * L * L
    pattern_bytes = nnz = 0
    if case["phase"] != "full":
        nb = L // case["block"]
        nnz = B * Hq * nb * sum(sd.sparsed_kept_per_row(_params(case), L))
        pattern_bytes = 4 * (B * Hq * nb + 1 + nnz)
    if case["phase"] == "select":
        side_bytes = (4 * B * Hq * L if case["lse"] else 0) + (4 * B * Hq * nb * nb if case["scores"] else 0)
        return {"bytes": q_bytes + kv_bytes + side_bytes + pattern_bytes, "flops": 2 * HEAD_DIM * logits}
    if case["phase"] == "sparse":
        return {"bytes": 2 * q_bytes + 2 * kv_bytes + pattern_bytes,
                "flops": 4 * HEAD_DIM * nnz * case["block"] * case["block"]}
    return {"bytes": 2 * q_bytes + 2 * kv_bytes + pattern_bytes, "flops": 4 * HEAD_DIM * logits}


def tolerance(case):
    # O: probabilities and outputs are rounded to bf16; measured 2.0e-3 to 2.2e-3 against 64 bits (1.66e-3 of it the
    # rounding of O alone), largest single difference 0.06 of the output's root mean square.
    # Block scores: fp32 sums of up to 16384 probabilities; measured 1.2e-6 between the two ways of taking them.
    # Selected lists: at the noise floor neighbouring scores lie a few 1e-8 apart, closer than two correct fp32 sums of
    # the same probabilities (those of the dense pass's row statistics and of a second Q K^T pass differ in up to 0.95 %
    # of the ids at 64k, 0.2 % at 8k), so a few ids change hands.
    if case["phase"] == "select":
        return {"rel": 5e-6, "differ": 1e-2}
    if case["phase"] == "switch":
        return {"rel": 1e-2, "differ": 1e-2}
    return {"rel": 1e-2}
