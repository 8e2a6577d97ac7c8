"""What a program that serves a diffusion language model has this library do, as measurable cases.

Every case is one pass through the public calls, in the order and with the arguments a serving loop uses, on one
stream and without host synchronisation.  Four kinds of pass:

  layers   one denoising step of the model's stack as a real model runs it, layer after layer: the window's Q/K/V
           projection with rotary embedding and the K/V rows staged in the cache, attention over [cache ; window], output
           projection.  Every layer has its own weights, hidden states and cache.
  stack    attention of all layers in one call (a caller that has every layer's Q/K/V up front).
  prefill  the initial full pass of a prompt: projection of all rows, attention with an empty cache, commit of the K/V
           rows; layer after layer.
  unmask   the sampling side of one block's life, from fully masked to filled: per step one pass over the vocabulary
           with the selection of positions, then, where the policy commits rows itself, the commit of the chosen rows.
           policy "topk": the k most confident positions; "entropy" / "margin" / "noise": ranked by another score;
           "guided": propose, accept the prefix an autoregressive guider agrees with, append the accepted rows;
           "guided_topk" / "guided_threshold": the other accept rules.

Values: hidden states, K/V and queries N(0, 1); weights N(0, 1 / K), so that projections are of unit scale; logits
sigma * N(0, 1) with sigma ~ U(1, 8) per position, so that confidences are skewed over the block.
"""
import math

import numpy as np
import torch

import paper_2505_21467_b200 as dlm

DEVICE = "cuda"
SCORES = {"entropy": dlm.DLM_SCORE_NEG_ENTROPY, "margin": dlm.DLM_SCORE_MARGIN, "noise": dlm.DLM_SCORE_LOG_CONF_PLUS_NOISE}
MAX_LOGIT_SETS = 8        # distinct logit tensors of a block's life (later steps cycle through them)
P_AGREE = 0.8             # the guider's token agrees with the proposal with this probability
TAU = 0.5                 # guidance confidence threshold

DREAM = dict(n_q_heads=28, n_kv_heads=4, head_dim=128, d_model=3584)
LLADA = dict(n_q_heads=32, n_kv_heads=32, head_dim=128, d_model=4096)
TINY = dict(n_q_heads=4, n_kv_heads=2, head_dim=64, d_model=256)
SMALL = dict(n_q_heads=8, n_kv_heads=2, head_dim=128, d_model=1024)
SMALL_MHA = dict(n_q_heads=8, n_kv_heads=8, head_dim=128, d_model=1024)
MODELS = [DREAM, LLADA, TINY, SMALL, SMALL_MHA]


def listed():
    return [
        # the smallest calls: one layer of the tiny configuration, three launches
        dict(name="tiny_step", kind="layers", layers=1, batch=1, block=32, cache=256, ragged=False, bias=False, **TINY),
        # interactive decoding, one sequence: a block of 32 behind a prompt of 1024, 28 layers
        dict(name="dream_step", kind="layers", layers=28, batch=1, block=32, cache=1024, ragged=False, bias=True, **DREAM),
        # the same stack recomputing the paper's window of 256 rows
        dict(name="dream_window_step", kind="layers", layers=28, batch=1, block=256, cache=1024, ragged=False, bias=True, **DREAM),
        # guided decoding of 8 sequences: prefix accepts leave every sequence with its own cache length and active rows
        dict(name="dream_batch8_step", kind="layers", layers=28, batch=8, block=32, cache=1152, ragged=True, bias=True, **DREAM),
        # multi-head stack, 4 sequences, block 64, prompt 2048, 32 layers
        dict(name="llada_step", kind="layers", layers=32, batch=4, block=64, cache=2048, ragged=False, bias=False, **LLADA),
        # attention of all 28 layers in one call, one sequence
        dict(name="dream_stack", kind="stack", layers=28, batch=1, block=32, cache=1024, ragged=False, **DREAM),
        # long context, cache length off the tile grid
        dict(name="long_context_stack", kind="stack", layers=28, batch=1, block=32, cache=16301, ragged=False, **DREAM),
        # the initial pass over prompt and generation area
        dict(name="dream_prefill", kind="prefill", layers=28, batch=1, block=1280, bias=True, **DREAM),
        # a block of 32 filled 4 positions per step, one sequence, chosen rows committed in every step
        dict(name="dream_topk_block", kind="unmask", policy="topk", batch=1, block=32, vocab=152064, k=4, layers=28, **DREAM),
        # blocks of 64 filled 4 positions per step by the entropy score, 4 sequences
        dict(name="llada_entropy_block", kind="unmask", policy="entropy", batch=4, block=64, vocab=126464, k=4, layers=0, **LLADA),
        # 8 sequences under the guided policy, 8 steps
        dict(name="dream_guided_block", kind="unmask", policy="guided", batch=8, block=32, vocab=152064, k=4, layers=28, **DREAM),
        # a vocabulary of odd size (rows not aligned to 16 bytes) and an odd block
        dict(name="odd_vocab_block", kind="unmask", policy="topk", batch=3, block=45, vocab=50021, k=5, layers=0, **SMALL),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    limit = 0.8 * max(_floor_s(c) for c in listed())
    while True:
        c = _draw_any(rng)
        if _floor_s(c) <= limit and _state_bytes(c) <= 10e9:
            return c


def _draw_any(rng):
    kind = rng.choice(["layers", "layers", "stack", "prefill", "unmask", "unmask"])
    model = rng.choice(MODELS)
    batch = _log_int(rng, 1, 8)
    if kind == "layers":
        # the output projection takes up to 256 rows, and whole groups of 8 per sequence when there are several
        block = _log_int(rng, 1, 256 // batch)
        if batch > 1:
            block = max(8, block // 8 * 8)
        return dict(kind=kind, layers=_log_int(rng, 1, 32), batch=batch, block=block, cache=_log_int(rng, 1, 4096),
                    ragged=batch > 1 and rng.random() < 0.5, bias=rng.random() < 0.5, **model)
    if kind == "stack":
        return dict(kind=kind, layers=_log_int(rng, 1, 32), batch=batch, block=_log_int(rng, 4, 512),
                    cache=_log_int(rng, 16, 20000), ragged=batch > 1 and rng.random() < 0.5, **model)
    if kind == "prefill":
        return dict(kind=kind, layers=_log_int(rng, 1, 28), batch=min(batch, 4), block=_log_int(rng, 32, 3000),
                    bias=rng.random() < 0.5, **model)
    policy = rng.choice(["topk", "topk", "entropy", "margin", "noise", "guided", "guided_topk", "guided_threshold"])
    return dict(kind=kind, policy=policy, batch=batch, block=_log_int(rng, 8, 128), vocab=_log_int(rng, 1000, 160000),
                k=rng.randint(1, 8), layers=rng.choice([0, 28]) if policy == "topk" else 28 if policy.startswith("guided") else 0,
                **model)


# ------------------------------------------------------------------------------------------------ sizes of a case

def _lengths(case):
    """(cache_len[b], q_len[b]) of a layers / stack case; a ragged batch has a spread of both, fixed by the case."""
    B, L, C = case["batch"], case["block"], case["cache"]
    if not case["ragged"]:
        return [C] * B, [L] * B
    return [max(1, C - (b * 53) % max(2, C // 4)) for b in range(B)], [max(1, L - (b * 5) % max(2, L * 3 // 4)) for b in range(B)]


def _steps(case):
    if case["policy"].startswith("guided"):
        return 8
    return -(-case["block"] // case["k"])


def _masked_rows(case):
    """Masked positions of one sequence that each step finds (guided: the expected number)."""
    L, left, rows = case["block"], float(case["block"]), []
    for s in range(_steps(case)):
        rows.append(left)
        if case["policy"].startswith("guided"):
            n = int(round(left))
            left -= min(left, sum(P_AGREE ** j for j in range(1, n + 1)) + (1 - P_AGREE if n else 0.0))
        else:
            left = max(0.0, L - (s + 1.0) * case["k"])
    return rows


def work(case):
    Hq, Hkv, D, dm = case["n_q_heads"], case["n_kv_heads"], case["head_dim"], case["d_model"]
    B, L, nl = case["batch"], case["block"], case["layers"]
    n_out, rows = (Hq + 2 * Hkv) * D, B * L
    if case["kind"] == "unmask":
        masked = sum(_masked_rows(case)) * B
        committed = B * L * (1 if nl else 0)
        return {"bytes": masked * case["vocab"] * 4 + committed * nl * Hkv * D * 2 * 2 * 2, "flops": masked * case["vocab"] * 3}
    if case["kind"] == "prefill":
        per_layer = 2 * n_out * dm + 2 * rows * dm + 4 * rows * D + 2 * rows * n_out    # weights, x, cos / sin, q / k / v
        per_layer += 2 * rows * Hq * D + 4 * rows * Hq + 4 * rows * Hkv * D             # attention output, lse, cache rows
        flops = 2 * rows * n_out * dm + 4 * B * Hq * L * L * D
        return {"bytes": nl * per_layer, "flops": nl * flops}
    lc, lq = _lengths(case)
    attn_bytes = 4 * Hkv * D * sum(c + q for c, q in zip(lc, lq)) + 2 * Hq * D * (sum(lq) + rows) + 4 * rows * Hq
    attn_flops = 4 * Hq * D * sum(q * (c + q) for c, q in zip(lc, lq))
    if case["kind"] == "stack":
        return {"bytes": nl * attn_bytes, "flops": nl * attn_flops}
    proj_bytes = 2 * n_out * dm + 2 * dm * Hq * D + 4 * rows * dm + 4 * rows * D + 2 * rows * n_out + 4 * Hkv * D * sum(lq)
    proj_flops = 2 * rows * n_out * dm + 2 * rows * dm * Hq * D
    return {"bytes": nl * (attn_bytes + proj_bytes), "flops": nl * (attn_flops + proj_flops)}


def _floor_s(case):
    w = work(case)
    return max(w["bytes"] / 6.5e12, w["flops"] / 1.6e15)


def _state_bytes(case):
    B, L, nl = case["batch"], case["block"], case["layers"]
    kv = 4 * nl * B * case["n_kv_heads"] * case["head_dim"]
    if case["kind"] == "unmask":
        return 4 * min(_steps(case), MAX_LOGIT_SETS) * B * L * case["vocab"] + 3 * kv * L
    return work(case)["bytes"] + kv * (L + case.get("cache", 0))


def tolerance(case):
    if case["kind"] == "unmask":
        # fp32 sums over the vocabulary in some order and an approximate exponential; tokens and positions are exact.  The
        # entropy is a difference of two sums that nearly cancel on flat rows.
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.0}
    # bf16 results (and, between the calls of a layer, bf16 intermediates) of fp32 sums
    return {"rel": 1e-2, "max": 0.1, "differ": 0.0}


# ------------------------------------------------------------------------------------------------ state

_context = None


def _ctx():
    """The process's library context, created once."""
    global _context
    if _context is None:
        _context = dlm.dlm_create(torch.cuda.current_device())
    return _context


class _Random:
    def __init__(self, seed):
        self.g = torch.Generator(device=DEVICE)
        self.g.manual_seed(int(seed))

    def bf16(self, *shape, scale=1.0):
        t = torch.empty(*shape, dtype=torch.bfloat16, device=DEVICE)
        return t.normal_(0.0, scale, generator=self.g)

    def uniform(self, *shape):
        return torch.rand(*shape, generator=self.g, device=DEVICE)


def _empty(*shape, dtype=torch.bfloat16):
    return torch.empty(*shape, dtype=dtype, device=DEVICE)


def _workspace(nbytes):
    return torch.empty(max(int(nbytes), 256), dtype=torch.uint8, device=DEVICE)


def _ints(values):
    return torch.tensor(values, dtype=torch.int32, device=DEVICE)


def _rope_tables(positions, D):
    """cos / sin of every (row, pair), fp32 [B][rows][D / 2]."""
    inv = torch.tensor(10000.0 ** (-np.arange(D // 2) * 2.0 / D), device=DEVICE)
    angle = positions[..., None].double() * inv
    return angle.cos().float().contiguous(), angle.sin().float().contiguous()


def prepare(case, seed):
    rnd, ctx = _Random(seed), _ctx()
    s = dict(case, ctx=ctx)
    Hq, Hkv, D, dm = case["n_q_heads"], case["n_kv_heads"], case["head_dim"], case["d_model"]
    B, L, nl = case["batch"], case["block"], case["layers"]
    n_out, rows = (Hq + 2 * Hkv) * D, B * L
    if case["kind"] == "unmask":
        return _prepare_unmask(s, rnd)
    if case["kind"] == "prefill":
        lc, lq = [0] * B, [L] * B
    else:
        lc, lq = _lengths(case)
    capacity = max(lc) + L
    s["k_cache"], s["v_cache"] = rnd.bf16(nl, B, Hkv, capacity, D), rnd.bf16(nl, B, Hkv, capacity, D)
    s["cache_len"] = _ints(lc)
    s["cache"] = dlm.make_kv_cache(s["k_cache"], s["v_cache"], s["cache_len"])
    s["hint"] = max(lc)
    s["q_len"] = _ints(lq) if case.get("ragged") else None
    n_call = nl if case["kind"] == "stack" else 1
    s["lse"] = _empty(nl, B, Hq, L, dtype=torch.float32)
    s["attn_ws"] = _workspace(dlm.dlm_attn_workspace_bytes(ctx, s["cache"], n_call, Hq, L))
    if case["kind"] == "stack":
        s["q"], s["k"], s["v"] = rnd.bf16(nl, B, Hq, L, D), rnd.bf16(nl, B, Hkv, L, D), rnd.bf16(nl, B, Hkv, L, D)
        s["o"] = _empty(nl, B, Hq, L, D)
        return s
    s["x"] = list(rnd.bf16(nl, B, L, dm))
    s["w_qkv"] = list(rnd.bf16(nl, n_out, dm, scale=dm ** -0.5))
    s["b_qkv"] = list(rnd.bf16(nl, n_out)) if case["bias"] else [None] * nl
    pos = torch.tensor(lc, device=DEVICE)[:, None] + torch.arange(L, device=DEVICE)[None, :]
    s["cos"], s["sin"] = _rope_tables(pos, D)
    # buffers of the activations between the calls, shared by the layers (the prefill keeps its layers' K/V apart)
    s["q"] = _empty(1, B, Hq, L, D)
    s["k"], s["v"] = _empty(1, B, Hkv, L, D), _empty(1, B, Hkv, L, D)
    s["o"] = _empty(nl, B, Hq, L, D)
    s["o_of"], s["lse_of"] = list(s["o"][:, None]), list(s["lse"][:, None])
    s["proj_ws"] = _workspace(max(dlm.dlm_window_proj_workspace_bytes(ctx, rows, n_out, dm),
                                  dlm.dlm_window_proj_workspace_bytes(ctx, rows, dm, Hq * D)))
    if case["kind"] == "layers":
        s["w_out"] = list(rnd.bf16(nl, dm, Hq * D, scale=(Hq * D) ** -0.5))
        s["y"] = _empty(nl, B, L, dm)
        s["y_of"] = list(s["y"])
    return s


def _prepare_unmask(s, rnd):
    B, L, V, k, nl = s["batch"], s["block"], s["vocab"], s["k"], s["layers"]
    n_steps = _steps(s)
    sets = min(n_steps, MAX_LOGIT_SETS)
    logits = torch.empty(sets, B, L, V, device=DEVICE).normal_(0.0, 1.0, generator=rnd.g)
    logits.mul_(1.0 + 7.0 * rnd.uniform(sets, B, L, 1))
    s["logits"] = list(logits)
    s["n_steps"] = n_steps
    s["masked"] = torch.ones(B, L, dtype=torch.uint8, device=DEVICE)
    s["tokens"] = torch.full((B, L), -1, dtype=torch.int32, device=DEVICE)
    s["tok"], s["conf"] = _empty(B, L, dtype=torch.int32), _empty(B, L, dtype=torch.float32)
    s["sel_idx"], s["n_sel"] = _empty(B, k, dtype=torch.int32), _empty(B, dtype=torch.int32)
    guided = s["policy"].startswith("guided")
    if s["policy"] in SCORES or s["policy"] == "guided_threshold":
        s["score"], s["zmax"] = _empty(B, L, dtype=torch.float32), _empty(B, L, dtype=torch.float32)
        u = rnd.uniform(B, L).clamp_(1e-6, 1.0 - 1e-6)
        s["noise"] = -(-u.log()).log() if s["policy"] == "noise" else None
        s["ws"] = _workspace(dlm.dlm_unmask_scored_workspace_bytes(s["ctx"], B, L, V))
    else:
        s["ws"] = _workspace(dlm.dlm_unmask_workspace_bytes(s["ctx"], B, L, V))
    if guided:
        top_k = 1 if s["policy"] == "guided" else 2
        best = torch.stack([z.max(dim=-1).indices for z in s["logits"]])                    # [sets][B][L]
        other = (best + 1 + (rnd.uniform(sets, B, L) * max(V - 2, 1)).long()) % V
        first = torch.where(rnd.uniform(sets, B, L) < P_AGREE, best, other)
        second = (first + 1) % V
        tok_ar = first[..., None] if top_k == 1 else torch.stack([first, second], dim=-1)
        s["top_k"], s["tok_ar"] = top_k, list(tok_ar.int().contiguous())
        if s["policy"] == "guided_threshold":
            s["logit_ar"] = list(20.0 + 40.0 * rnd.uniform(sets, B, L, top_k))
        s["accept"] = _empty(B, L, dtype=torch.uint8)
        s["acc_idx"], s["n_acc"] = _empty(B, L, dtype=torch.int32), _empty(B, dtype=torch.int32)
    if nl:
        capacity = 64 + L
        s["k_cache"], s["v_cache"] = rnd.bf16(nl, B, s["n_kv_heads"], capacity, s["head_dim"]), rnd.bf16(nl, B, s["n_kv_heads"], capacity, s["head_dim"])
        s["k_new"], s["v_new"] = rnd.bf16(nl, B, s["n_kv_heads"], L, s["head_dim"]), rnd.bf16(nl, B, s["n_kv_heads"], L, s["head_dim"])
        s["cache_len"] = _ints([64] * B)
        s["cache"] = dlm.make_kv_cache(s["k_cache"], s["v_cache"], s["cache_len"])
    return s


# ------------------------------------------------------------------------------------------------ one pass

def run(s):
    return {"layers": _run_layers, "stack": _run_stack, "prefill": _run_prefill, "unmask": _run_unmask}[s["kind"]](s)


def _run_layers(s):
    ctx, cache, B, L, dm = s["ctx"], s["cache"], s["batch"], s["block"], s["d_model"]
    Hq, Hkv, D = s["n_q_heads"], s["n_kv_heads"], s["head_dim"]
    q, k, v = s["q"], s["k"], s["v"]
    for l in range(s["layers"]):
        dlm.dlm_window_qkv_project_stage(ctx, s["x"][l], s["w_qkv"][l], s["b_qkv"][l], s["cos"], s["sin"], B, L, dm, Hq, Hkv, D,
                                         s["q_len"], q, k, v, cache, l, s["proj_ws"])
        dlm.dlm_freecache_attn_step(ctx, cache, l, l + 1, q, k, v, Hq, L, s["q_len"], 0.0, s["hint"], s["o_of"][l], s["lse_of"][l],
                                    s["attn_ws"])
        dlm.dlm_window_out_project(ctx, s["o_of"][l], s["w_out"][l], None, B, L, dm, Hq, D, s["y_of"][l], s["proj_ws"])
    return {"y": s["y"], "o": s["o"], "lse": s["lse"], "q": q, "k": k, "v": v, "k_cache": s["k_cache"], "v_cache": s["v_cache"]}


def _run_stack(s):
    dlm.dlm_freecache_attn_step(s["ctx"], s["cache"], 0, s["layers"], s["q"], s["k"], s["v"], s["n_q_heads"], s["block"], s["q_len"],
                                0.0, s["hint"], s["o"], s["lse"], s["attn_ws"])
    return {"o": s["o"], "lse": s["lse"]}


def _run_prefill(s):
    ctx, cache, B, L, nl = s["ctx"], s["cache"], s["batch"], s["block"], s["layers"]
    Hq, Hkv, D = s["n_q_heads"], s["n_kv_heads"], s["head_dim"]
    q, k, v = s["q"], s["k"], s["v"]
    s["cache_len"].zero_()
    for l in range(nl):
        dlm.dlm_window_qkv_project_rope(ctx, s["x"][l], s["w_qkv"][l], s["b_qkv"][l], s["cos"], s["sin"], B, L, s["d_model"], Hq, Hkv, D,
                                        q, k, v, s["proj_ws"])
        dlm.dlm_freecache_attn_step(ctx, cache, l, l + 1, q, k, v, Hq, L, None, 0.0, 1, s["o_of"][l], s["lse_of"][l], s["attn_ws"])
        dlm.dlm_kv_cache_commit(ctx, cache, k, v, L, None, None, dlm.DLM_DST_APPEND, None, L, l == nl - 1, l, l + 1)
    return {"o": s["o"], "lse": s["lse"], "q": q, "k_cache": s["k_cache"], "v_cache": s["v_cache"], "cache_len": s["cache_len"]}


def _run_unmask(s):
    ctx, B, L, V, k, nl, policy = s["ctx"], s["batch"], s["block"], s["vocab"], s["k"], s["layers"], s["policy"]
    masked, tokens, tok, conf, ws = s["masked"], s["tokens"], s["tok"], s["conf"], s["ws"]
    out = {"tok": tok, "conf": conf, "masked": masked, "tokens": tokens}
    masked.fill_(1)
    tokens.fill_(-1)
    if nl:
        s["cache_len"].fill_(64)
        out.update(k_cache=s["k_cache"], v_cache=s["v_cache"], cache_len=s["cache_len"])
    for step in range(s["n_steps"]):
        i = step % len(s["logits"])
        z = s["logits"][i]
        if policy in SCORES:
            dlm.dlm_unmask_select_scored(ctx, z, B, L, V, masked, tokens, k, SCORES[policy], s["noise"], tok, conf, s["score"], s["zmax"],
                                         s["sel_idx"], s["n_sel"], ws)
        elif policy == "topk":
            dlm.dlm_unmask_select(ctx, z, B, L, V, masked, tokens, k, tok, conf, s["sel_idx"], s["n_sel"], ws)
            if nl:      # the rows chosen in this step go to their own slots behind the visible ones
                dlm.dlm_kv_cache_commit(ctx, s["cache"], s["k_new"], s["v_new"], L, s["sel_idx"], None, dlm.DLM_DST_WINDOW, s["n_sel"], k,
                                        0, 0, nl)
        else:
            if policy == "guided_threshold":
                dlm.dlm_unmask_select_scored(ctx, z, B, L, V, masked, tokens, 0, dlm.DLM_SCORE_CONFIDENCE, None, tok, conf, s["score"],
                                             s["zmax"], None, None, ws)
                dlm.dlm_guided_accept_threshold(ctx, tok, s["zmax"], s["tok_ar"][i], s["logit_ar"][i], s["top_k"], TAU, B, L, masked, tokens,
                                                0, s["accept"], s["acc_idx"], s["n_acc"])
            else:
                dlm.dlm_unmask_select(ctx, z, B, L, V, masked, tokens, 0, tok, conf, None, None, ws)
                if policy == "guided":
                    dlm.dlm_guided_accept(ctx, tok, s["tok_ar"][i], B, L, masked, tokens, 0, s["accept"], s["acc_idx"], s["n_acc"])
                else:
                    dlm.dlm_guided_accept_topk(ctx, tok, s["tok_ar"][i], s["top_k"], B, L, masked, tokens, 0, s["accept"], s["acc_idx"],
                                               s["n_acc"])
            if nl:      # the accepted rows become visible at once
                dlm.dlm_kv_cache_commit(ctx, s["cache"], s["k_new"], s["v_new"], L, s["acc_idx"], None, dlm.DLM_DST_APPEND, s["n_acc"], L, 1, 0, nl)
    if policy.startswith("guided"):
        out.update(accept=s["accept"], acc_idx=s["acc_idx"], n_acc=s["n_acc"])
    else:
        out.update(sel_idx=s["sel_idx"], n_sel=s["n_sel"])
    if policy in SCORES or policy == "guided_threshold":
        out.update(score=s["score"], zmax=s["zmax"])
    return out
