"""What a user of this library has it do, as cases whose speed can be measured: whole calls of the step loop
(`Engine.prefill` and `Engine.step`) from one interactive question to a serving batch, and the stand-alone decode
attention at the cache sizes that the step loop reaches only after hours of decoding.

`listed()` names the cases, `draw(rng)` gives others of the same ranges, `prepare(case, seed)` builds models, prompts
and engine on the GPU, `run(state)` makes one pass, `work(case)` counts what such a pass cannot do without and
`tolerance(case)` says how far another correct implementation of the same precision may be off.

Shapes are those of the repository's configurations (fp32 test pair, small bf16 pair, 1.5B / 7B / 72B decoders).  Where
full depth would not fit the GPU three times over or a pass would take too long, the depth is cut and nothing else:
every layer of a model runs the same kernels on the same shapes.

The models are random but behave like trained ones in the two respects that decide what the step loop does.  Their
next-token distributions are peaked: the head maps a token's own embedding to a fixed successor, drawn as a
permutation, so that sampling at the paper's temperatures is all but deterministic; draft and target agree on 85 % of
the successors.  The PRM's scores are bimodal: its embedding carries a good / bad direction, 70 % of the tokens are
good, and the layers spread the scores around two modes on either side of the threshold.  So the token streams and the
gate decisions have margins far above rounding, and one changed rounding does not send two correct implementations
down different paths; the rewards and the logits depend on every layer.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2501_19324_b200 import Engine, Model, RSD_DEBUG_KEEP_LOGITS
from paper_2501_19324_b200.binding import k_attn_decode

# layers, width, query heads, KV heads, head dim, FFN width, vocabulary
SHAPES = {
    "tiny_draft": (2, 256, 4, 2, 64, 688, 1024),
    "tiny_target": (4, 512, 8, 2, 64, 1376, 1024),
    "mini_draft": (2, 512, 4, 2, 128, 1408, 4096),
    "mini_target": (3, 768, 6, 2, 128, 2048, 4096),
    "1.5b": (28, 1536, 12, 2, 128, 8960, 151936),
    "7b": (28, 3584, 28, 4, 128, 18944, 151936),
    "72b": (80, 8192, 64, 8, 128, 29568, 152064),
}
GOOD_SHARE = 0.7     # share of tokens the PRM likes: about the accept rate of the paper's runs
AGREE_SHARE = 0.85   # share of tokens whose successor draft and target agree on
CLASS_WEIGHT = 0.15  # good / bad component of the PRM's embedding, in units of an embedding entry


def _step(name, draft, prm, target, batch, lo, hi, cap, steps, **more):
    """A pass: prefill `batch` prompts of lo..hi tokens, then `steps` calls of Engine.step with steps of at most `cap`
    tokens.  depth_*: layers kept (0 = all).  end_mod: one token in end_mod ends its step (0 = one id of the vocabulary
    does: nearly every step runs to the cap).  min_rows > 1: queued rejections.  sd: proposals of a speculative round.  merged: the PRM is
    a head on the draft.  ext: hi + lo KV cache.  chunk: tokens of a multi-token pass (0 = the library's default)."""
    case = dict(kind="step", draft=draft, prm=prm, target=target, batch=batch, lo=lo, hi=hi, cap=cap, steps=steps,
                depth_draft=0, depth_prm=0, depth_target=0, end_mod=0, temperature=0.7, delta=0.7, min_rows=1, sd=0,
                merged=False, ext=0, chunk=0, logits=False, device_outputs=False)
    case.update(more)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # the fp32 models of the smallest configuration, as it stands: 4 rows, 4 greedy steps that end at id 13 or at 32
        # tokens.  All latency: a model fits a corner of the chip.
        _step("fp32-4rows", "tiny_draft", "tiny_draft", "tiny_target", 4, 64, 64, 32, 4, temperature=0.0),
        # a small bf16 model pair, ragged prompts and steps: launches and host time of the 16-bit path
        _step("small-bf16-8rows", "mini_draft", "mini_draft", "mini_target", 8, 32, 96, 16, 4, end_mod=16),
        # one interactive question on the 1.5B / 1.5B / 7B models, a few reasoning steps: decode at one row
        _step("one-question", "1.5b", "1.5b", "7b", 1, 128, 512, 32, 4, end_mod=32),
        # three rows whose caller wants the logits of every generated token (log-probabilities) beside the tokens
        _step("logits-3rows", "1.5b", "1.5b", "7b", 3, 33, 129, 8, 2, logits=True),
        # the headline workload at full depth: 32 rows, prompts of 128..512 tokens; the second step syncs the draft
        # and scores target-written tokens as all later ones do
        _step("paper-32rows", "1.5b", "1.5b", "7b", 32, 128, 512, 64, 2, end_mod=64, chunk=8192),
        # PRM at the target's shape, 64 rows of 256-token prompts; half the depth
        _step("wide-prm-64rows", "1.5b", "7b", "7b", 64, 256, 256, 48, 2, depth_draft=14, depth_prm=14, depth_target=14,
              chunk=8192),
        # a target of the 72B shape, cut to 12 layers, with the hi + lo cache that its full depth takes
        _step("large-target-8rows", "1.5b", "1.5b", "72b", 8, 256, 256, 32, 1, depth_draft=14, depth_prm=14,
              depth_target=12, ext=1),
        # long documents: prefill, scoring and catch-up attention over thousands of cached tokens, then decode over them
        _step("long-prompts", "1.5b", "1.5b", "7b", 5, 4000, 8000, 24, 1, depth_draft=14, depth_prm=14, depth_target=14),
        # a serving batch whose rejected rows wait until 16 of them share a target pass
        _step("queued-40rows", "1.5b", "1.5b", "7b", 40, 100, 200, 24, 4, depth_draft=14, depth_prm=14, depth_target=14,
              end_mod=24, min_rows=16),
        # rejected steps rewritten by speculative decoding: four proposals a round
        _step("speculative-16rows", "1.5b", "1.5b", "7b", 16, 128, 256, 32, 2, depth_draft=14, depth_prm=14,
              depth_target=14, sd=4, temperature=0.0),
        # the largest batch: 128 short rows, the PRM a head on the draft, results left on the GPU
        _step("merged-128rows", "1.5b", "1.5b", "7b", 128, 48, 128, 24, 2, depth_draft=14, depth_prm=14, depth_target=14,
              merged=True, device_outputs=True),
        # decode attention alone at a long-running batch: 64 rows with ragged contexts of up to 16384 tokens
        dict(name="decode-attention-64x16k", kind="attn", batch=64, ctx_lo=4096, ctx_hi=16384, heads=28, kv_heads=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["tiny", "mini", "paper", "paper", "wide", "large", "long", "attn"])
    if family == "attn":
        heads, kv = rng.choice([(12, 2), (28, 4), (64, 8)])
        hi = _log_int(rng, 512, 16384)
        return dict(kind="attn", batch=_log_int(rng, 1, 256 if hi * kv <= 16384 else 64), ctx_lo=rng.randint(1, hi),
                    ctx_hi=hi, heads=heads, kv_heads=kv)
    temperature = rng.choice([0.0, 0.7])
    hi = _log_int(rng, 32, {"tiny": 96, "large": 384}.get(family, 512))
    lo = rng.randint(max(1, hi // 4), hi)
    cap = _log_int(rng, 6, 40)
    end_mod = rng.choice([0, cap, 2 * cap])
    if family == "tiny":
        return _step("", "tiny_draft", "tiny_draft", "tiny_target", rng.randint(1, 8), lo, hi, cap, rng.randint(1, 4),
                     temperature=temperature, end_mod=end_mod)
    if family == "mini":
        return _step("", "mini_draft", "mini_draft", "mini_target", _log_int(rng, 1, 64), lo, hi, cap, rng.randint(1, 4),
                     temperature=temperature, end_mod=end_mod, sd=rng.choice([0, 0, 3]), ext=rng.choice([0, 0, 1]))
    depth = rng.randint(4, 14)
    more = dict(depth_draft=depth, depth_prm=depth, depth_target=depth, temperature=temperature, end_mod=end_mod)
    if family == "long":
        hi = _log_int(rng, 1000, 8000)
        return _step("", "1.5b", "1.5b", "7b", max(1, min(8, 30000 // hi)), hi // 2, hi, cap, 1, **more)
    if family == "large":
        more["depth_target"] = rng.randint(2, 12)
        return _step("", "1.5b", "1.5b", "72b", rng.randint(1, 12), lo, hi, cap, 1, ext=rng.choice([0, 1]), **more)
    batch = min(_log_int(rng, 1, 96), 16384 // hi)
    steps = rng.randint(1, 2)
    if family == "wide":
        return _step("", "1.5b", "7b", "7b", batch, lo, hi, cap, steps, **more)
    option = rng.choice(["plain", "plain", "queue", "sd", "merged"])
    if option == "queue":
        more["min_rows"] = max(2, batch // 3)
    if option == "sd" and batch <= 32:
        more["sd"] = rng.choice([2, 4, 7])
    return _step("", "1.5b", "1.5b", "7b", batch, lo, hi, cap, steps, merged=option == "merged", **more)


# ---- models ------------------------------------------------------------------------------------------------------

def _shape(case, role):
    layers, d, H, KV, hd, F, V = SHAPES[case[role]]
    return SimpleNamespace(n_layers=case["depth_" + role] or layers, d_model=d, n_heads=H, n_kv_heads=KV, head_dim=hd,
                           d_ffn=F, vocab=V, rope_theta=1.0e4, rms_eps=1.0e-6)


def _layers_rms(sh):
    """Root mean square of what the layers add to an entry of the residual stream.  The MLPs add nearly all of it: a gate
    or up value is N(0, (0.02 sqrt(d))^2) and the down projection sums d_ffn products silu(gate) up."""
    var = 0.0004 * sh.d_model
    g = np.linspace(-6, 6, 1001) * math.sqrt(var)
    p = np.exp(-0.5 * g * g / var)
    silu_sq = float(((g / (1 + np.exp(-g))) ** 2 * p).sum() / p.sum())
    return math.sqrt(sh.n_layers * 0.0004 * sh.d_ffn * silu_sq * var)


def _tensors(sh, dtype, gen):
    """Layer weights N(0, 0.02) and norm gains 1 +- 0.1; an embedding as large as what the layers add to it; no head yet."""
    def normal(*size, std=0.02):
        return torch.randn(*size, generator=gen, device="cuda", dtype=dtype).mul_(std)

    def gain():
        return (1 + 0.1 * torch.rand(sh.d_model, generator=gen, device="cuda").mul(2).sub(1)).to(dtype)

    d, hq, hkv, F = sh.d_model, sh.n_heads * sh.head_dim, sh.n_kv_heads * sh.head_dim, sh.d_ffn
    t = dict(tok_embed=normal(sh.vocab, d, std=_layers_rms(sh)), final_norm=gain(), wqkv=[], wo=[], wgu=[], wdown=[],
             norm1=[], norm2=[])
    for _ in range(sh.n_layers):
        t["wqkv"].append(normal(hq + 2 * hkv, d))
        t["wo"].append(normal(d, hq))
        t["wgu"].append(normal(2 * F, d))
        t["wdown"].append(normal(d, F))
        t["norm1"].append(gain())
        t["norm2"].append(gain())
    return t


def _lm_head(sh, embed, successor):
    """Head whose row successor[v] is the embedding of v, scaled so that the successor's logit is about 30: the final
    hidden state, embedding plus layers over their common rms, has 1 / sqrt(2) of the embedding in it."""
    head = torch.zeros_like(embed)
    head[successor] = embed[: successor.numel()] * (30.0 * math.sqrt(2.0) / (sh.d_model * _layers_rms(sh)))
    return head


def _add_classes(sh, embed, good, gen):
    """Adds the good / bad direction to an embedding; returns the PRM head that reads it, scores about +-3.4."""
    w = torch.randint(0, 2, (sh.d_model,), generator=gen, device="cuda").mul_(2).sub_(1).to(embed.dtype)
    embed[: good.numel()] += (CLASS_WEIGHT * _layers_rms(sh) * (good.to(embed.dtype) * 2 - 1))[:, None] * w
    return w * (3.4 * math.sqrt(2.0) / (CLASS_WEIGHT * sh.d_model))


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(1000003 * seed + 17)
    if case["kind"] == "attn":
        return _prepare_attn(case, gen, seed)
    dtype = torch.float32 if case["draft"].startswith("tiny") else torch.bfloat16
    sd, sp, st = (_shape(case, r) for r in ("draft", "prm", "target"))
    v = min(sd.vocab, sp.vocab, st.vocab)
    successor = torch.randperm(v, generator=gen, device="cuda")
    # the target's successors: the draft's with 15 % of them moved on in a ring
    moved = torch.nonzero(torch.rand(v, generator=gen, device="cuda") >= AGREE_SHARE).flatten()
    successor_t = successor.clone()
    successor_t[moved] = successor[moved.roll(1)]
    good = torch.rand(v, generator=gen, device="cuda") < GOOD_SHARE

    draft = _tensors(sd, dtype, gen)
    prm = draft if case["merged"] else _tensors(sp, dtype, gen)
    prm = dict(prm, head=_add_classes(sp, prm["tok_embed"], good, gen))
    draft = dict(draft, head=_lm_head(sd, draft["tok_embed"], successor))
    target = _tensors(st, dtype, gen)
    target["head"] = _lm_head(st, target["tok_embed"], successor_t)

    models = (Model(sd, draft, 0), Model(sp, prm, 1, head_only=case["merged"]), Model(st, target, 0))
    eng = Engine(*models, max_batch=case["batch"], max_seq_tokens=case["hi"] + (case["steps"] + 1) * case["cap"],
                 max_step_tokens=case["cap"], max_steps=case["steps"] + 1, step_end_id=13, step_end_mod=case["end_mod"],
                 temperature=case["temperature"], seed=seed % 1000, max_chunk_tokens=case["chunk"],
                 debug_flags=RSD_DEBUG_KEEP_LOGITS if case["logits"] else 0, kv_extended=case["ext"],
                 prm_shares_draft=int(case["merged"]), sd_tokens=case["sd"])
    rng = np.random.default_rng(seed)
    lens = rng.integers(case["lo"], case["hi"] + 1, size=case["batch"])
    offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    tokens = rng.integers(0, v, size=int(offsets[-1])).astype(np.int32)
    return dict(case=case, engine=eng, tokens=tokens, offsets=offsets)


def _prepare_attn(case, gen, seed):
    """A fp16 paged cache whose pages are handed out in no particular order, as after many rows have come and gone."""
    B, H, KV, hd = case["batch"], case["heads"], case["kv_heads"], 128
    rng = np.random.default_rng(seed)
    ctx = rng.integers(case["ctx_lo"], case["ctx_hi"] + 1, size=B).astype(np.int32)
    max_pages = (case["ctx_hi"] + 15) // 16
    pool = torch.randn(B * max_pages, 2 * KV * 16 * hd, generator=gen, device="cuda", dtype=torch.float16)
    table = torch.randperm(B * max_pages, generator=gen, device="cuda").to(torch.int32).view(B, max_pages)
    q = torch.randn(B, H, hd, generator=gen, device="cuda")
    return dict(case=case, q=q, pool=pool, table=table, ctx=torch.from_numpy(ctx).cuda())


def run(state):
    case = state["case"]
    if case["kind"] == "attn":
        return k_attn_decode(state["q"], state["pool"], state["table"], state["ctx"], case["kv_heads"])
    eng = state["engine"]
    eng.prefill(state["tokens"], state["offsets"])
    step = eng.step_device if case["device_outputs"] else eng.step
    out = []
    for _ in range(case["steps"]):
        r = step(case["delta"], case["min_rows"])
        if case["logits"]:
            # the draft's for every row, the target's for the rows that it wrote
            r["draft_logits"], r["target_logits"] = eng.logits(0), eng.logits(2)
            r["target_logits"][r["accept"] == 1] = 0
        out.append(r)
    return {"steps": out, "counters": eng.counters()}


# ---- what a pass cannot do without -------------------------------------------------------------------------------

def _params(sh, head):
    d, hd, H, KV, F = sh.d_model, sh.head_dim, sh.n_heads, sh.n_kv_heads, sh.d_ffn
    return sh.n_layers * (2 * d * H * hd + 2 * d * KV * hd + 3 * d * F) + (sh.vocab * d if head else 0)


def _iterations(rows, case):
    """(Expected length of the longest, expected length of one) of `rows` steps."""
    p = 1.0 / (case["end_mod"] or SHAPES[case["draft"]][6])
    longest = sum(1 - (1 - (1 - p) ** j) ** rows for j in range(case["cap"]))
    return longest, sum((1 - p) ** j for j in range(case["cap"]))


def work(case):
    """Bytes: each model's weights once per decode iteration and once per multi-token pass, the cached keys and values
    that an iteration attends.  Flops: two per parameter and token, four per head dim and attended position.  Step
    lengths and accept rate enter with their expected values."""
    if case["kind"] == "attn":
        ctx, B, hd = 0.5 * (case["ctx_lo"] + case["ctx_hi"]), case["batch"], 128
        return {"bytes": B * (ctx * 2 * case["kv_heads"] * hd * 2 + 2 * case["heads"] * hd * 4), "flops": 4.0 * B * ctx * case["heads"] * hd}
    B, elem = case["batch"], 4 if case["draft"].startswith("tiny") else 2
    sd, sp, st = (_shape(case, r) for r in ("draft", "prm", "target"))
    prompt = 0.5 * (case["lo"] + case["hi"])
    bytes_ = flops = 0.0

    def kv(sh):
        return sh.n_layers * 2 * sh.n_kv_heads * sh.head_dim * (4 if case["ext"] else elem)

    def attn(sh):
        return 4.0 * sh.n_layers * sh.n_heads * sh.head_dim

    def dense(sh, tokens, ctx):
        nonlocal bytes_, flops
        bytes_ += _params(sh, False) * elem + tokens * kv(sh)
        flops += tokens * (2.0 * _params(sh, False) + attn(sh) * ctx)

    def decode(sh, iters, rows, mean_len, ctx):
        nonlocal bytes_, flops
        bytes_ += iters * _params(sh, True) * elem + rows * mean_len * ctx * kv(sh)
        flops += rows * mean_len * (2.0 * _params(sh, True) + attn(sh) * ctx)

    dense(sd, B * prompt, prompt / 2)
    if not case["merged"]:
        dense(sp, B * prompt, prompt / 2)
    rejected = (1 - GOOD_SHARE) * B
    some = 1 - GOOD_SHARE ** B                                   # probability that a step rejects any row
    for k in range(case["steps"]):
        longest, mean = _iterations(B, case)
        ctx = prompt + k * mean
        decode(sd, longest, B, mean, ctx)
        if case["merged"]:
            decode(sd, 1, B, 1, ctx)
        else:
            dense(sp, B * mean, ctx)
        longest, mean = _iterations(max(1, round(rejected)), case)
        rounds = longest / (1 + AGREE_SHARE * (case["sd"] - 1)) if case["sd"] else longest
        share = some if case["min_rows"] <= 1 else min(1.0, rejected / case["min_rows"])
        if k == 0 or share < 1:
            dense(st, share * rejected * prompt, prompt / 2)
        decode(st, share * rounds, share * rejected, mean, ctx)
        if case["sd"]:
            decode(sd, share * longest, share * rejected, mean, ctx)
    if case["logits"]:
        bytes_ += case["steps"] * B * case["cap"] * (sd.vocab + (1 - GOOD_SHARE) * st.vocab) * 4
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """About four times what was seen between the path and itself with hi + lo operands and caches throughout (16-bit
    models: rewards up to rel 5e-4, max 8e-4; logits below that)."""
    if case["kind"] == "attn":
        # fp16 queries and softmax weights, fp32 sums
        return {"rel": 1.5e-3, "max": 1e-2}
    if case["draft"].startswith("tiny"):
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.0}
    return {"rel": 2.5e-3, "max": 1e-2, "differ": 0.002}
