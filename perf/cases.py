"""The work whose speed matters to a user of this library, as measurable cases.

A serving loop of speculative decoding calls one verify step per emitted block (attention of the block rows over the
paged cache, LM head + acceptance, commit of the lengths) and, on the drafter's side, one single-row step or one nucleus
draw per proposed token; an alignment run adds the total variation distance of every drafted position.  ``listed`` names
points of these, ``draw`` takes more of the same ranges:

  step    massv_verify_attn + massv_accept + massv_kv_commit through ``VerifyStep`` (batch 1 .. 64, gamma 0 .. 7, greedy and
          sampling, contexts of a few positions up to 32k, head dims 64 / 128 / 256, vocabularies of 1k .. 262k); ``host``
          takes the inputs from pinned host memory and the result back (``VerifyStep.run_host``); ``probs`` asks for the
          dense distribution as well (the drafter's own step: gamma 0, the row it samples from is the q of the next verify step)
  attn    massv_verify_attn alone: what every layer but the last adds to a step, here with the sliding window of local layers
  top_p   massv_sample_top_p over rows of logits
  tvd     massv_tvd of drafted positions

Values: K, V, Q ~ N(0, 1) in bf16, pages scattered over the pool.  The hidden states are scaled so that logits have a
standard deviation of 5 (the largest of 152k probabilities is then 0.1 - 0.5, as a language model's are); the drafter's
logits are the target's plus N(0, 1).
"""
import math
import random

import torch

from paper_2505_10526_b200 import VerifyStep
from paper_2505_10526_b200 import binding as mv

PAGE = 16
DEV = "cuda"
LOGIT_STD = 5.0

_QWEN = dict(q_heads=28, kv_heads=4, head_dim=128, hidden=3584, vocab=152064)
_GEMMA = dict(q_heads=16, kv_heads=8, head_dim=256, hidden=3840, vocab=262144)
_TINY = dict(q_heads=4, kv_heads=1, head_dim=64, hidden=256, vocab=1024)
_DRAFTER = dict(q_heads=12, kv_heads=2, head_dim=128, hidden=1536, vocab=152064)


def _step(shape, batch, gamma, temperature, ctx_lo, ctx_hi, host=False, probs=False):
    return dict(kind="step", batch=batch, gamma=gamma, **shape, temperature=float(temperature), ctx_lo=ctx_lo, ctx_hi=ctx_hi,
                window=0, host=host, probs=probs)


def _attn(shape, batch, gamma, ctx_lo, ctx_hi, window):
    return dict(kind="attn", batch=batch, gamma=gamma, q_heads=shape["q_heads"], kv_heads=shape["kv_heads"],
                head_dim=shape["head_dim"], ctx_lo=ctx_lo, ctx_hi=ctx_hi, window=window)


def listed():
    return [
        # the smallest call: launches and the host path are all there is
        dict(name="tiny_b1_t1", **_step(_TINY, 1, 5, 1.0, 256, 256)),
        # one user, greedy, an image prompt of 1,280 positions: the latency of one emitted block
        dict(name="qwen7b_b1_t0", **_step(_QWEN, 1, 5, 0.0, 1280, 1280)),
        # a few users at the start of their answers: odd batch, short ragged contexts, another gamma and temperature
        dict(name="qwen7b_b7_g3_t07", **_step(_QWEN, 7, 3, 0.7, 1, 777)),
        # eight greedy users whose step inputs come from the host and whose tokens go back there
        dict(name="qwen7b_b8_t0_host", **_step(_QWEN, 8, 5, 0.0, 512, 2048, host=True)),
        # a server's ordinary batch at the paper's sampling settings
        dict(name="qwen7b_b16_t1", **_step(_QWEN, 16, 5, 1.0, 1024, 4096)),
        # the other target shape: head dim 256, a vocabulary of 262,144
        dict(name="gemma12b_b32_t1", **_step(_GEMMA, 32, 5, 1.0, 2048, 8192)),
        # a local layer of that target (five of six layers look like this): window of 1,024 positions
        dict(name="gemma12b_b32_local", **_attn(_GEMMA, 32, 5, 2048, 8192, 1024)),
        # the largest batch over long contexts, sampling
        dict(name="qwen7b_long_g5_t1", **_step(_QWEN, 64, 5, 1.0, 8192, 32768)),
        # and greedy with the longest block: 512 rows through the LM head
        dict(name="qwen7b_long_g7_t0", **_step(_QWEN, 64, 7, 0.0, 8192, 32768)),
        # the drafter's own step for the ordinary batch: one row per sequence, its distribution is the next step's q
        dict(name="drafter_b16_t1", **_step(_DRAFTER, 16, 0, 1.0, 1024, 4096, probs=True)),
        # nucleus sampling of the same rows for a batch of 64 (self-distillation responses, a sampling drafter)
        dict(name="top_p_b64", kind="top_p", rows=64, vocab=152064, temperature=1.0, top_p=0.9, probs=True),
        # the alignment diagnostic over a batch of 64 blocks
        dict(name="tvd_b64_g5", kind="tvd", batch=64, gamma=5, vocab=152064, temperature=1.0),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def _draw_shape(rng):
    pick = rng.randrange(5)
    if pick < 2:
        return dict(_QWEN)
    if pick == 2:
        return dict(_GEMMA)
    kv = rng.choice((1, 2, 4, 8))
    return dict(q_heads=kv * rng.randint(1, 8), kv_heads=kv, head_dim=rng.choice((64, 128, 256)),
                hidden=64 * _log_int(rng, 4, 64), vocab=8 * _log_int(rng, 128, 20000))


def _draw_context(rng):
    hi = _log_int(rng, 16, 32768)
    return rng.randint(min(hi, max(1, hi // 4)), hi), hi


def draw(rng):
    largest = [max(x) for x in zip(*[(w["bytes"], w["flops"]) for w in map(work, listed())])]
    while True:
        kind = rng.choice(("step",) * 6 + ("attn", "attn", "top_p", "tvd"))
        if kind in ("step", "attn"):
            shape = _draw_shape(rng)
            lo, hi = _draw_context(rng)
            batch, gamma = _log_int(rng, 1, 64), rng.randint(0, 7)
            if shape["q_heads"] // shape["kv_heads"] * (gamma + 1) > 64 or batch * (gamma + 1) > 512:
                continue
            if kind == "attn":
                case = _attn(shape, batch, gamma, lo, hi, rng.choice((0, 0, 512, 1024)))
            else:
                temperature = rng.choice((0.0, 0.7, 1.0))
                case = _step(shape, batch, gamma, temperature, lo, hi, host=temperature == 0.0 and rng.random() < 0.25,
                             probs=temperature > 0 and rng.random() < (0.75 if gamma == 0 else 0.1))
        elif kind == "top_p":
            case = dict(kind="top_p", rows=_log_int(rng, 1, 256), vocab=8 * _log_int(rng, 128, 32768), temperature=rng.choice((0.6, 0.8, 1.0)),
                        top_p=rng.choice((0.8, 0.9, 0.95, 1.0)), probs=rng.random() < 0.75)
        else:
            case = dict(kind="tvd", batch=_log_int(rng, 1, 64), gamma=rng.randint(1, 7), vocab=8 * _log_int(rng, 128, 32768),
                        temperature=rng.choice((0.7, 1.0)))
        w = work(case)
        if w["bytes"] <= largest[0] and w["flops"] <= largest[1]:
            return case


# ---------------------------------------------------------------- inputs
def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _attention_inputs(case, seed, gen):
    B, R = case["batch"], case["gamma"] + 1
    kv, d = case["kv_heads"], case["head_dim"]
    r = random.Random(seed)
    lens = [r.randint(case["ctx_lo"], case["ctx_hi"]) for _ in range(B)]
    max_pages = -(-(case["ctx_hi"] + R) // PAGE)
    used = [-(-(n + R) // PAGE) for n in lens]
    n_pages = B * max_pages                       # the pool does not depend on the lengths
    ids = torch.randperm(n_pages, generator=gen, device=DEV, dtype=torch.int32).cpu()
    table = torch.full((B, max_pages), -1, dtype=torch.int32)
    at = 0
    for b, n in enumerate(used):
        table[b, :n] = ids[at:at + n]
        at += n
    bf = dict(dtype=torch.bfloat16, device=DEV, generator=gen)
    return dict(q=torch.randn((B, R, case["q_heads"], d), **bf), k_new=torch.randn((B, R, kv, d), **bf), v_new=torch.randn((B, R, kv, d), **bf),
                k_pages=torch.randn((n_pages, kv, PAGE, d), **bf), v_pages=torch.randn((n_pages, kv, PAGE, d), **bf),
                page_table=table.to(DEV), seq_lens=torch.tensor(lens, dtype=torch.int32, device=DEV))


def _drafter(logits, temperature, gen):
    """The drafter's distribution and its tokens for rows of target logits [B, gamma, V]."""
    zq = logits + torch.randn(logits.shape, generator=gen, device=DEV)
    if temperature == 0:
        return None, zq.argmax(dim=-1).to(torch.int32)
    q = torch.softmax(zq / temperature, dim=-1)
    # one exponential race per row: argmax of q / Exp(1) is a draw from q
    race = torch.empty_like(q).exponential_(generator=gen)
    return q, (q / race).argmax(dim=-1).to(torch.int32)


def _accept_inputs(case, gen):
    B, g, K, V = case["batch"], case["gamma"], case["hidden"], case["vocab"]
    R = g + 1
    std = LOGIT_STD / (0.02 * math.sqrt(K))
    out = dict(hidden=(torch.randn((B, R, K), device=DEV, generator=gen) * std).to(torch.bfloat16),
               lm_head=torch.randn((V, K), device=DEV, dtype=torch.bfloat16, generator=gen).mul_(0.02))
    z = torch.matmul(out["hidden"].view(B * R, K), out["lm_head"].t()).float().view(B, R, V)
    q, tokens = (None, torch.zeros((B, 0), dtype=torch.int32, device=DEV)) if g == 0 else _drafter(z[:, :g], case["temperature"], gen)
    out["draft_tokens"] = tokens.contiguous()
    if case["temperature"] > 0:
        out["draft_probs"] = q.contiguous() if q is not None else torch.zeros((B, 0, V), device=DEV)
        out["u_accept"] = torch.rand((B, g), device=DEV, generator=gen)
        out["u_sample"] = torch.rand((B, R), device=DEV, generator=gen)
    return out


def _inputs(case, seed):
    gen = _generator(seed)
    if case["kind"] in ("step", "attn"):
        w = _attention_inputs(case, seed, gen)
        if case["kind"] == "step":
            w.update(_accept_inputs(case, gen))
        return w
    if case["kind"] == "top_p":
        return dict(logits=LOGIT_STD * torch.randn((case["rows"], case["vocab"]), device=DEV, generator=gen),
                    u=torch.rand((case["rows"],), device=DEV, generator=gen))
    B, g, V = case["batch"], case["gamma"], case["vocab"]
    z = LOGIT_STD * torch.randn((B, g + 1, V), device=DEV, generator=gen)
    return dict(logits=z, draft_probs=_drafter(z[:, :g], case["temperature"], gen)[0].contiguous())


def prepare(case, seed):
    w = _inputs(case, seed)
    state = dict(case=case, w=w)
    if case["kind"] == "step":
        step = VerifyStep(case["batch"], case["gamma"], case["q_heads"], case["kv_heads"], case["head_dim"], case["hidden"], case["vocab"],
                          case["temperature"], w["page_table"].shape[1], w["k_pages"].shape[0], device=DEV, window=case["window"],
                          want_logits=True, want_probs=case["probs"])
        state["step"] = step
        # the lengths the next step would start from: a buffer of their own, so that a pass can be run again on the same cache
        state["next_lens"] = w["seq_lens"].clone()
        if case["host"]:
            per_step = {k: w.pop(k) for k in ("q", "k_new", "v_new", "hidden", "draft_tokens")}
            state["host_inputs"] = step.host_inputs_like(per_step)
    elif case["kind"] == "attn":
        state["desc"] = mv.attn_desc(case["batch"], case["gamma"], case["q_heads"], case["kv_heads"], case["head_dim"],
                                     w["page_table"].shape[1], w["k_pages"].shape[0], window=case["window"])
        state["ws"] = mv.alloc_workspace(mv.massv_verify_attn_workspace_size(state["desc"]), DEV)
        state["out"] = torch.empty_like(w["q"])
        state["status"] = torch.zeros((1,), dtype=torch.int32, device=DEV)
    elif case["kind"] == "top_p":
        state["tokens"] = torch.empty((case["rows"],), dtype=torch.int32, device=DEV)
        state["probs"] = torch.empty_like(w["logits"]) if case["probs"] else None
        state["status"] = torch.zeros((1,), dtype=torch.int32, device=DEV)
    else:
        state["desc"] = mv.accept_desc(case["batch"], case["gamma"], 64, case["vocab"], case["temperature"])
        state["ws"] = mv.alloc_workspace(mv.massv_tvd_workspace_size(state["desc"]), DEV)
        state["tvd"] = torch.empty((case["batch"], case["gamma"]), device=DEV)
        state["accept_prob"] = torch.empty_like(state["tvd"])
        state["status"] = torch.zeros((1,), dtype=torch.int32, device=DEV)
    return state


def run(state):
    case, w = state["case"], state["w"]
    if case["kind"] == "step":
        step = state["step"]
        if case["host"]:
            tokens, lens = step.run_host(state["host_inputs"], w)
        else:
            step.run(w, commit=False)
            tokens, lens = step.out_tokens, step.accept_len
        step.commit(state["next_lens"])
        return dict(attn=step.attn_out, k_pages=w["k_pages"], v_pages=w["v_pages"], logits=step.logits, probs=step.probs, tokens=tokens,
                    accept_len=lens, next_lens=state["next_lens"], status=step.dev_status)
    if case["kind"] == "attn":
        mv.massv_verify_attn(state["desc"], w["q"], w["k_new"], w["v_new"], w["k_pages"], w["v_pages"], w["page_table"], w["seq_lens"],
                             state["out"], None, None, state["ws"], state["status"])
        return dict(attn=state["out"], k_pages=w["k_pages"], v_pages=w["v_pages"], status=state["status"])
    if case["kind"] == "top_p":
        mv.massv_sample_top_p(w["logits"], w["u"], state["tokens"], case["temperature"], case["top_p"], state["probs"], state["status"])
        return dict(tokens=state["tokens"], probs=state["probs"], status=state["status"])
    mv.massv_tvd(state["desc"], w["logits"], w["draft_probs"], state["tvd"], state["accept_prob"], state["ws"], state["status"])
    return dict(tvd=state["tvd"], accept_prob=state["accept_prob"], status=state["status"])


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    if case["kind"] == "top_p":
        n = case["rows"] * case["vocab"]
        return dict(bytes=n * (8 if case["probs"] else 4), flops=4.0 * n)
    if case["kind"] == "tvd":
        n = case["batch"] * case["gamma"] * case["vocab"]
        return dict(bytes=8 * n, flops=8.0 * n)
    B, R, d, hq, hkv = case["batch"], case["gamma"] + 1, case["head_dim"], case["q_heads"], case["kv_heads"]
    ctx = (case["ctx_lo"] + case["ctx_hi"]) / 2
    seen = min(ctx, case["window"] - 1) if case["window"] else ctx
    nbytes = 4.0 * B * (seen + 2 * R) * hkv * d + 4.0 * B * R * hq * d            # cache and block K/V, the block's slots; q and out
    flops = 4.0 * B * R * hq * d * (seen + R / 2)
    if case["kind"] == "step":
        M, K, V = B * R, case["hidden"], case["vocab"]
        nbytes += 2.0 * V * K + 2.0 * M * K + 4.0 * M * V                          # weights, hidden states, logits
        flops += 2.0 * M * V * K
        if case["temperature"] > 0 and case["gamma"] > 0:
            nbytes += 4.0 * B * V                                                  # the drafter's row at the rejection
        if case["probs"]:
            nbytes += 4.0 * M * V
    return dict(bytes=nbytes, flops=flops)


def tolerance(case):
    # tvd, top_p: fp32 exponentials.  Attention leaves in bf16 after softmax weights in bf16; logits are fp32 sums of bf16 products.
    if case["kind"] in ("tvd", "top_p"):
        return {"rel": 1e-5, "max": 1e-3, "differ": 0.0}
    return {"rel": 1e-2, "max": 0.1, "differ": 0.0}


# ---------------------------------------------------------------- the same in 64 bits
def _exact_attention(case, w):
    B, R, d, hkv = case["batch"], case["gamma"] + 1, case["head_dim"], case["kv_heads"]
    G = case["q_heads"] // hkv
    out = torch.empty((B, R, case["q_heads"], d), dtype=torch.float64, device=DEV)
    for b, n in enumerate(w["seq_lens"].tolist()):
        pages = w["page_table"][b, :-(-n // PAGE)].long()
        first = 0 if not case["window"] else max(0, n - case["window"] + 1)          # the earliest position a row sees
        k, v = (torch.cat([w[p][pages].transpose(0, 1).reshape(hkv, -1, d)[:, first:n], w[x][b].transpose(0, 1)], dim=1).double()
                for p, x in (("k_pages", "k_new"), ("v_pages", "v_new")))
        q = w["q"][b].double().view(R, hkv, G, d).permute(1, 0, 2, 3).reshape(hkv, R * G, d)
        s = torch.matmul(q, k.transpose(1, 2)) / math.sqrt(d)
        pos = torch.arange(first, n + R, device=DEV)
        row = n + torch.arange(R, device=DEV).repeat_interleave(G)
        hidden = pos[None, :] > row[:, None]
        if case["window"]:
            hidden |= pos[None, :] <= row[:, None] - case["window"]
        s.masked_fill_(hidden[None], -math.inf)
        o = torch.matmul(torch.softmax(s, dim=-1), v)
        out[b] = o.view(hkv, R, G, d).permute(1, 0, 2, 3).reshape(R, case["q_heads"], d)
    return out


def _exact_logits(w):
    B, R, K = w["hidden"].shape
    h = w["hidden"].view(B * R, K).double()
    V = w["lm_head"].shape[0]
    z = torch.empty((B * R, V), dtype=torch.float64, device=DEV)
    for v in range(0, V, 32768):
        z[:, v:v + 32768] = torch.matmul(h, w["lm_head"][v:v + 32768].double().t())
    return z.view(B, R, V)


def exact(case, seed):
    w = _inputs(case, seed)
    if case["kind"] == "attn":
        return dict(attn=_exact_attention(case, w), k_pages=None, v_pages=None, status=None)
    if case["kind"] == "step":
        z = _exact_logits(w)
        return dict(attn=_exact_attention(case, w), k_pages=None, v_pages=None, logits=z,
                    probs=torch.softmax(z / case["temperature"], dim=-1) if case["probs"] else None, tokens=None, accept_len=None,
                    next_lens=None, status=None)
    if case["kind"] == "top_p":
        if not case["probs"]:
            return None
        p = torch.softmax(w["logits"].double() / case["temperature"], dim=-1)
        top, at = torch.sort(p, dim=-1, descending=True, stable=True)
        before = torch.cumsum(top, dim=-1) - top
        kept = torch.zeros_like(p).scatter_(-1, at, torch.where(before < case["top_p"], top, 0.0))
        return dict(tokens=None, probs=kept / kept.sum(dim=-1, keepdim=True), status=None)
    B, g = case["batch"], case["gamma"]
    p = torch.softmax(w["logits"][:, :g].double() / case["temperature"], dim=-1)
    q = w["draft_probs"].double()
    return dict(tvd=0.5 * (p - q).abs().sum(dim=-1), accept_prob=torch.minimum(p, q).sum(dim=-1), status=None)
