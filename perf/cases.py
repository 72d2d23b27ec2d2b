"""What a user of the verification step runs, as cases that can be timed and compared.

A case names one call of the public interface (`entry`) and the shape of the batch it is called on:

  attention  wisp_verify_attention: the k + 1 new queries of each request over its paged KV cache
  accept     wisp_verify_accept: the lossless acceptance pass over the vocabulary
  greedy     wisp_verify_accept_greedy: its temperature-0 variant
  step       wisp_verify_step: attention and acceptance in one call
  round      wisp_kv_reserve_append, wisp_verify_step, wisp_kv_commit: one served batch

Lengths follow from the case alone (so that every seed does the same amount of work); the order of
the requests, every tensor and the page placement follow from the seed.  Values are those of a served
batch: Q, K, V ~ N(0, 1), logits ~ N(0, 2), draft distributions softmax(logits + noise) with the noise
that gives each request's acceptance rate, draft tokens drawn from them, uniform random numbers.
"""
import math

import numpy as np
import torch

from paper_2601_11652_gb300 import binding as wb

PAGE = 16
DEV = "cuda"


# ------------------------------------------------------------------------------------------ cases
def _case(name, entry, *, B, heads=(32, 8, 128), dtype="bf16", k=(1, 8), ctx=(512, 4096), long_share=0.0, long=(0, 0),
          law="uniform", V=128256, alpha=(0.7, 0.7), shuffle=False):
    c = {"entry": entry, "B": B, "Hq": heads[0], "Hkv": heads[1], "D": heads[2], "dtype": dtype, "k_lo": k[0], "k_hi": k[1],
         "ctx_law": law, "ctx_lo": ctx[0], "ctx_hi": ctx[1], "long_share": long_share, "long_lo": long[0],
         "long_hi": long[1], "V": V, "alpha_lo": alpha[0], "alpha_hi": alpha[1], "shuffle": shuffle}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest call: a handful of short fp32 requests on a small vocabulary (a test or a toy
        # model); launches and latency count
        _case("step_tiny_f32", "step", B=4, heads=(4, 4, 64), dtype="f32", k=(1, 4), ctx=(16, 128), V=1000),
        # one request alone, as a lightly loaded server sees it
        _case("attention_b1", "attention", B=1, k=(4, 4), ctx=(4096, 4096)),
        # an ordinary batch of a serving engine: the whole verification of one layer
        _case("step_b32", "step", B=32),
        # many edge devices at once: ragged short and medium contexts, drafts of up to 16 tokens
        _case("attention_b256", "attention", B=256, k=(1, 16), law="lognormal", ctx=(1, 16384)),
        # few requests with very long contexts on a fragmented page pool
        _case("attention_long_b16", "attention", B=16, k=(4, 8), ctx=(32768, 131072), shuffle=True),
        # a small model's heads of 64 with plain decode requests (k = 0) among the drafts
        _case("attention_d64_b64", "attention", B=64, heads=(32, 8, 64), k=(0, 8), ctx=(256, 8192), shuffle=True),
        # the ordinary batch with an fp32 cache (a reference run, or a model kept in fp32)
        _case("attention_f32_b32", "attention", B=32, dtype="f32"),
        # the acceptance pass on its own, as an engine calls it whose attention runs inside the model
        _case("accept_b256", "accept", B=256, k=(1, 16), alpha=(0.4, 0.9)),
        # ... with fp32 logits (an engine that keeps its head's output in fp32) and a larger vocabulary
        _case("accept_f32_b16", "accept", B=16, dtype="f32", k=(0, 8), V=152064),
        # temperature 0
        _case("greedy_b256", "greedy", B=256, k=(1, 16), alpha=(0.4, 0.9)),
        # one round of the serving loop: pages and new K/V rows, the step, the commit
        _case("round_b64", "round", B=64, heads=(28, 4, 128), k=(0, 12), ctx=(256, 1024), long_share=0.3,
              long=(8192, 32768), V=152064, alpha=(0.3, 0.95)),
        # the largest: short and long requests with and without drafts, a full server
        _case("step_b512", "step", B=512, heads=(28, 4, 128), k=(0, 12), ctx=(256, 1024), long_share=0.3,
              long=(8192, 32768), V=152064, alpha=(0.3, 0.95)),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    entry = rng.choice(["attention", "attention", "accept", "greedy", "step", "step", "round"])
    dtype = "f32" if rng.random() < 0.2 else "bf16"
    heads = rng.choice([(32, 8, 128), (28, 4, 128), (8, 2, 128), (32, 8, 64), (8, 2, 64), (4, 4, 64)])
    g = heads[0] // heads[1]
    B = _log_int(rng, 1, 512 if dtype == "bf16" else 32)
    k_hi = rng.randint(0, min(16, 128 // g - 1))
    k_lo = rng.randint(0, k_hi)
    token = 2 * heads[1] * heads[2] * (2 if dtype == "bf16" else 4)  # KV bytes of a token
    most = min(131072, int((4e9 if dtype == "bf16" else 4e8) / (B * token)))
    hi = _log_int(rng, 32, max(64, most))
    V = min(_log_int(rng, 1000, 152064), int(2.5e9 / (B * (k_hi + 1) * 6)))  # logits and draft rows: 2.5 GB at most
    if rng.random() < 0.75:  # most vocabularies are padded to a multiple of 64, some are not
        V = (V + 63) // 64 * 64
    a = rng.uniform(0.3, 0.95)
    return _case(None, entry, B=B, heads=heads, dtype=dtype, k=(k_lo, k_hi), ctx=(max(1, hi // rng.choice([1, 2, 8, 32])), hi),
                 law=rng.choice(["uniform", "lognormal"]), V=V, alpha=(a, min(0.95, a + 0.3)), shuffle=rng.random() < 0.5)


def _lengths(c):
    """Draft and context lengths of the batch: of the case alone."""
    r = np.random.default_rng([c["B"], c["k_hi"], c["ctx_hi"], c["D"], 7])
    B = c["B"]
    k = r.integers(c["k_lo"], c["k_hi"] + 1, B)
    if c["ctx_law"] == "lognormal":
        mid = max(1.0, c["ctx_hi"] / 8)
        ctx = np.clip(np.round(r.lognormal(math.log(mid), 1.0, B)), c["ctx_lo"], c["ctx_hi"]).astype(np.int64)
    else:
        ctx = r.integers(c["ctx_lo"], c["ctx_hi"] + 1, B)
    if c["long_share"] > 0:
        far = r.random(B) < c["long_share"]
        ctx = np.where(far, r.integers(c["long_lo"], c["long_hi"] + 1, B), ctx)
    return k.astype(np.int64), ctx.astype(np.int64)


# ------------------------------------------------------------------------------------------ inputs
def _inputs(c, seed):
    """Every tensor of the case on the GPU, and the lengths on the host (request order of the seed)."""
    k, ctx = _lengths(c)
    host = np.random.default_rng([int(seed), 11])
    order = host.permutation(c["B"])
    k, ctx = k[order], ctx[order]
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) * 1000003 + 17)
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    B, Tq, Td = c["B"], int(k.sum()) + c["B"], int(k.sum())
    i32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).to(DEV)  # noqa: E731

    def normal(shape, sd=1.0):
        x = torch.randn(shape, generator=gen, device=DEV, dtype=dt)
        return x if sd == 1.0 else x.mul_(sd)

    t = {"draft_lens": i32(k), "request_ids": torch.arange(1000, 1000 + B, dtype=torch.int64, device=DEV)}
    if c["entry"] in ("attention", "step", "round"):
        nblk = (ctx + k + 1 + PAGE - 1) // PAGE
        have = (ctx + PAGE - 1) // PAGE if c["entry"] == "round" else nblk  # pages a request brings along
        num = int(nblk.sum()) + (64 if c["entry"] == "round" else 0)
        ids = host.permutation(num) if c["shuffle"] else np.arange(num)
        bt = np.full((B, int(nblk.max())), -1, dtype=np.int32)
        at = 0
        for r in range(B):
            bt[r, :have[r]] = ids[at:at + have[r]]
            at += int(have[r])
        t["context_lens"], t["block_tables"] = i32(ctx), i32(bt)
        t["q"] = normal((Tq, c["Hq"], c["D"]))
        t["k_cache"] = normal((num, c["Hkv"], PAGE, c["D"]))
        t["v_cache"] = normal((num, c["Hkv"], PAGE, c["D"]))
        t["out"] = torch.empty_like(t["q"])
        if c["entry"] == "round":
            free = np.concatenate([ids[at:], np.zeros(at, ids.dtype)])  # the stack; entries past the count are unused
            t["free_blocks"], t["free_count"] = i32(free), i32([num - at])
            t["k_new"], t["v_new"] = normal((Tq, c["Hkv"], c["D"])), normal((Tq, c["Hkv"], c["D"]))
    if c["entry"] != "attention":
        V = c["V"]
        alpha = torch.from_numpy(host.uniform(c["alpha_lo"], c["alpha_hi"], B)).to(DEV)
        sigma = 2.0 * math.sqrt(2.0) * torch.special.erfinv(1.0 - alpha)
        t["logits"] = normal((Tq, V), 2.0)
        row = np.concatenate([np.arange(n) + s for n, s in zip(k, np.cumsum(k + 1) - (k + 1))]) if Td else np.zeros(0)
        row = torch.from_numpy(row.astype(np.int64)).to(DEV)
        sig = torch.repeat_interleave(sigma, torch.from_numpy(k).to(DEV)).float()
        t["draft_probs"] = torch.empty((Td, V), dtype=torch.float32, device=DEV)
        t["draft_tokens"] = torch.empty(Td, dtype=torch.int32, device=DEV)
        for a in range(0, Td, 256):
            b = min(Td, a + 256)
            x = torch.randn((b - a, V), generator=gen, device=DEV).mul_(sig[a:b, None]).add_(t["logits"][row[a:b]].float())
            qd = torch.softmax(x, dim=1)
            t["draft_probs"][a:b] = qd
            # a token drawn from the distribution: the largest q / Exp(1)
            t["draft_tokens"][a:b] = (qd / torch.empty_like(qd).exponential_(generator=gen)).argmax(dim=1).int()
        if c["entry"] == "greedy":  # a draft that agrees with the target's choice as often as its acceptance rate
            best = t["logits"][row].argmax(dim=1).int() if Td else t["draft_tokens"]
            agree = torch.rand(Td, generator=gen, device=DEV) < torch.repeat_interleave(alpha, torch.from_numpy(k).to(DEV))
            t["draft_tokens"] = torch.where(agree, best, t["draft_tokens"]).contiguous()
        t["accept_u"] = torch.rand(Td, generator=gen, device=DEV)
        t["sample_u"] = torch.rand(B, generator=gen, device=DEV)
        t["accepted_len"] = torch.full((B,), -7, dtype=torch.int32, device=DEV)
        t["next_token"] = torch.full((B,), -7, dtype=torch.int32, device=DEV)
    return t, k, ctx


def prepare(case, seed):
    t, k, _ = _inputs(case, seed)
    e = case["entry"]
    s = {"entry": e, "t": t}
    if e in ("attention", "step", "round"):
        s["attn"] = wb.make_attn_args(draft_lens=t["draft_lens"], context_lens=t["context_lens"],
                                      block_tables=t["block_tables"], q=t["q"], k_cache=t["k_cache"],
                                      v_cache=t["v_cache"], out=t["out"], request_ids=t["request_ids"])
    if e != "attention":
        s["acc"] = wb.make_accept_args(draft_lens=t["draft_lens"], target_logits=t["logits"],
                                       draft_tokens=t["draft_tokens"], draft_probs=t["draft_probs"],
                                       accept_uniforms=t["accept_u"], sample_uniforms=t["sample_u"],
                                       accepted_len=t["accepted_len"], next_token=t["next_token"],
                                       request_ids=t["request_ids"])
    s["ws"] = wb.alloc_workspace(wb.wisp_verify_workspace_size(s.get("attn"), s.get("acc")), DEV)
    if e == "round":
        s["kv"] = wb.make_kv_args(draft_lens=t["draft_lens"], context_lens=t["context_lens"],
                                  block_tables=t["block_tables"], free_blocks=t["free_blocks"],
                                  free_count=t["free_count"], k_cache=t["k_cache"], v_cache=t["v_cache"],
                                  k_new=t["k_new"], v_new=t["v_new"], accepted_len=t["accepted_len"],
                                  request_ids=t["request_ids"], total_q_rows=int(k.sum()) + case["B"])
        s["kvws"] = wb.alloc_workspace(wb.wisp_kv_workspace_size(s["kv"]), DEV)
        s["sessions"] = {n: t[n].clone() for n in ("context_lens", "block_tables", "free_blocks", "free_count")}
    return s


def run(s):
    e, t = s["entry"], s["t"]
    if e == "attention":
        wb.wisp_verify_attention(s["attn"], s["ws"])
        return t["out"]
    if e == "accept":
        wb.wisp_verify_accept(s["acc"], s["ws"])
        return {"accepted_len": t["accepted_len"], "next_token": t["next_token"]}
    if e == "greedy":
        wb.wisp_verify_accept_greedy(s["acc"], s["ws"])
        return {"accepted_len": t["accepted_len"], "next_token": t["next_token"]}
    if e == "step":
        wb.wisp_verify_step(s["attn"], s["acc"], s["ws"])
        return {"out": t["out"], "accepted_len": t["accepted_len"], "next_token": t["next_token"]}
    # the batch's rows of the session tables, as the serving loop gathers them before each round
    for n, v in s["sessions"].items():
        t[n].copy_(v)
    wb.wisp_kv_reserve_append(s["kv"], s["kvws"])
    wb.wisp_verify_step(s["attn"], s["acc"], s["ws"])
    wb.wisp_kv_commit(s["kv"], s["kvws"])
    return {n: t[n] for n in ("out", "accepted_len", "next_token", "context_lens", "block_tables", "free_blocks",
                              "free_count", "k_cache", "v_cache")}


# ------------------------------------------------------------------------------------------ cost
def work(case):
    k, ctx = _lengths(case)
    e, es = case["entry"], 2 if case["dtype"] == "bf16" else 4
    Tq, V = int(k.sum()) + case["B"], case["V"]
    by = fl = 0.0
    if e in ("attention", "step", "round"):
        n = ctx + k + 1
        by += float(n.sum()) * case["Hkv"] * case["D"] * 2 * es  # K and V of every visible token
        by += Tq * case["Hq"] * case["D"] * 2 * es               # queries and outputs
        by += 4.0 * float(((n + PAGE - 1) // PAGE).sum())
        fl += 4.0 * case["D"] * case["Hq"] * float(((k + 1) * (ctx + 1) + k * (k + 1) // 2).sum())
    if e != "attention":
        # logit rows 0..L (the rule stops at the first rejection); L is random: its mean at the case's
        # acceptance rate.  After a rejection one draft row as well.
        a = 0.5 * (case["alpha_lo"] + case["alpha_hi"])
        rows = float(sum((1 - a ** (int(x) + 1)) / (1 - a) for x in k))
        by += rows * V * es + 72.0 * rows
        fl += 4.0 * rows * V
        if e != "greedy":
            by += float(sum(1 - a ** int(x) for x in k)) * V * 4
    if e == "round":
        by += 2.0 * Tq * case["Hkv"] * case["D"] * 2 * es                       # the new rows: read and written
        by += 4.0 * float(((ctx + k + 1 + PAGE - 1) // PAGE).sum())             # the table entries looked at
    return {"bytes": by, "flops": fl}


def tolerance(case):
    if case["entry"] in ("accept", "greedy"):
        return "exact"
    # bf16: P and the output are rounded to 8 bits (2.3e-3 measured against 64 bits); fp32: 32-bit sums
    return {"rel": 1e-2, "max": 0.2, "differ": 0.0} if case["dtype"] == "bf16" else {"rel": 4e-6, "max": 1e-4, "differ": 0.0}


# ------------------------------------------------------------------------------------------ 64 bits
def _exact_attention(c, t, k, ctx, bt):
    out = torch.empty(t["q"].shape, dtype=torch.float64, device=DEV)
    g, at = c["Hq"] // c["Hkv"], 0
    for r in range(c["B"]):
        n, m = int(ctx[r] + k[r] + 1), int(k[r] + 1)
        pages = bt[r, :(n + PAGE - 1) // PAGE].long()
        q = t["q"][at:at + m].double().view(m, c["Hkv"], g, c["D"]).transpose(0, 1)       # [Hkv, m, g, D]
        kk = t["k_cache"][pages].transpose(0, 1).reshape(c["Hkv"], -1, c["D"])[:, :n].double()
        s = torch.matmul(q.reshape(c["Hkv"], m * g, c["D"]), kk.transpose(1, 2)) / math.sqrt(c["D"])
        seen = torch.arange(n, device=DEV)[None, :] <= (int(ctx[r]) + torch.arange(m, device=DEV))[:, None]
        s = s.view(c["Hkv"], m, g, n).masked_fill(~seen[None, :, None, :], -math.inf).softmax(dim=-1)
        del kk
        vv = t["v_cache"][pages].transpose(0, 1).reshape(c["Hkv"], -1, c["D"])[:, :n].double()
        o = torch.matmul(s.view(c["Hkv"], m * g, n), vv).view(c["Hkv"], m, g, c["D"])
        out[at:at + m] = o.transpose(0, 1).reshape(m, c["Hq"], c["D"])
        at += m
    return out


def _exact_accept(c, t, k):
    L, tok = torch.empty(c["B"], dtype=torch.int32), torch.empty(c["B"], dtype=torch.int32)
    q0 = d0 = 0
    for r in range(c["B"]):
        m = int(k[r])
        z = t["logits"][q0:q0 + m + 1].double()
        y = t["draft_tokens"][d0:d0 + m].long()
        if c["entry"] == "greedy":
            best = z.argmax(dim=1)
            ok = (best[:m] == y).long()
            n = int(ok.cumprod(0).sum())
            nxt = int(best[n])
        else:
            p = torch.softmax(z, dim=1)
            qy = t["draft_probs"][torch.arange(d0, d0 + m, device=DEV), y].double()
            py = p[torch.arange(m, device=DEV), y]
            a = torch.where(qy == 0, torch.ones_like(qy), torch.clamp(py / qy, max=1.0))
            ok = (t["accept_u"][d0:d0 + m].double() <= a).long()
            n = int(ok.cumprod(0).sum())
            w = p[n]
            if n < m:
                res = torch.clamp(w - t["draft_probs"][d0 + n].double(), min=0.0)
                w = res if float(res.sum()) > 0 else w
            cdf = w.cumsum(0)
            hit = cdf > t["sample_u"][r].double() * cdf[-1]
            nxt = int(hit.int().argmax()) if bool(hit.any()) else int(w.nonzero()[-1])
        L[r], tok[r] = n, nxt
        q0, d0 = q0 + m + 1, d0 + m
    return L, tok


def exact(case, seed):
    t, k, ctx = _inputs(case, seed)
    e = case["entry"]
    if e == "attention":
        return _exact_attention(case, t, k, ctx, t["block_tables"])
    if e in ("accept", "greedy"):
        L, tok = _exact_accept(case, t, k)
        return {"accepted_len": L, "next_token": tok}
    if e == "step":
        L, tok = _exact_accept(case, t, k)
        return {"out": _exact_attention(case, t, k, ctx, t["block_tables"]), "accepted_len": L, "next_token": tok}
    # round: pages from the top of the free stack in request order, the new rows, the step, the commit
    bt, ctx_h = t["block_tables"].cpu().numpy().copy(), ctx.copy()
    free = t["free_blocks"].cpu().numpy().copy()
    count, at, before = int(t["free_count"].item()), 0, bt
    for r in range(case["B"]):
        for b in range(int(-(-(ctx[r] + k[r] + 1) // PAGE))):
            if bt[r, b] < 0:
                count -= 1
                bt[r, b] = free[count]
        for j in range(int(k[r]) + 1):
            pos = int(ctx[r]) + j
            t["k_cache"][bt[r, pos // PAGE], :, pos % PAGE] = t["k_new"][at]
            t["v_cache"][bt[r, pos // PAGE], :, pos % PAGE] = t["v_new"][at]
            at += 1
    out = _exact_attention(case, t, k, ctx, torch.from_numpy(before).to(DEV))
    L, tok = _exact_accept(case, t, k)
    for r in range(case["B"]):
        new = int(ctx[r]) + 1 + int(L[r])
        for b in range(-(-new // PAGE), int(-(-(ctx[r] + k[r] + 1) // PAGE))):
            if bt[r, b] >= 0:
                free[count], bt[r, b] = bt[r, b], -1
                count += 1
        ctx_h[r] = new
    return {"out": out, "accepted_len": L, "next_token": tok, "context_lens": torch.from_numpy(ctx_h.astype(np.int32)),
            "block_tables": torch.from_numpy(bt), "free_blocks": torch.from_numpy(free),
            "free_count": torch.tensor([count], dtype=torch.int32), "k_cache": t["k_cache"], "v_cache": t["v_cache"]}
