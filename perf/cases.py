"""Performance cases: the work a user of the verify-step library has it do.

Every case goes through the package's public entry points, the way a serving
or training program calls them: buffers, workspaces and (where the program
would keep one) a CUDA graph are made once in `prepare`; `run` is one pass.

Kinds of case
  step    a whole verify step (attention of both caches, vocabulary pass with
          the verdict, loss) through VerifyStep: issued call by call, replayed
          from a captured graph, or fed from pinned host memory
  attn    ipd.verify_attn with the proposers' decode in the same launch, or
          ipd.decode_attn alone (the proposal phase between two verify steps)
  score   ipd.score_span_ex with other rules, by-products and the next draw
  train   top-K lists, the split loss and its gradient (the backward pass)
  kl      ipd.full_kl, the monitoring pass
  sample  ipd.sample, the proposers' draw of one token per row
  append  ipd.kv_append_many, a step's new K/V rows into both caches

Shapes are the Qwen3-like pair of this repository's workloads: teacher 32
query / 4 KV heads, student 16 / 8, head_dim 128, pages of 16 tokens placed at
random in the pools, K/V/Q ~ N(0, 1); logits N(0, sigma^2), "boost" (the
verifier's logit of the proposed token raised so that about 60 % are covered)
or "zipf".  Context and span lengths are the quantiles of a case's distribution,
assigned to requests at random, so that inputs of another seed are other
inputs of the same total size.
"""
import math

import torch

from paper_2609_36546_gb300 import VerifyStep, ipd

PAGE, D = 16, 128
HEADS = {"t": (32, 4), "s": (16, 8)}  # query / KV heads of teacher and student
SCALE = 1.0 / math.sqrt(128.0)
QWEN_VOCAB = 151936
TOKEN_OUTS = ("logp_s", "logp_t", "feedback", "kl_rev", "kl_fwd")
TAU = 3.0  # entropy threshold of the "entropy" rules, nats
SAMPLE_SEED = 0x5EED


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _case(name, kind, requests, ctx, span=(4, 4), **kw):
    c = {"kind": kind, "requests": requests, "ctx_lo": ctx[0], "ctx_hi": ctx[1],
         "ctx_median": ctx[2] if len(ctx) > 2 else 0,  # > 0: lognormal (sigma 1), clipped
         "span_lo": span[0], "span_hi": span[1], "direction": "half", "vocab": QWEN_VOCAB,
         "logits": "boost", "K": 16}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one interactive user's step: four short requests over a small
        # vocabulary, issued call by call; launches and host time are all of it
        _case("step tiny", "step", 4, (64, 256), vocab=4096, logits="normal", how="calls",
              rows="all"),
        # the everyday serving step: 64 student-driven requests, span 8, replayed
        # from a graph
        _case("step 64", "step", 64, (1024, 8192), (8, 8), direction="S",
              how="graph", rows="all"),
        # the full rollout step: 1024 requests, ragged spans, both drivers, only
        # the needed logits rows read
        _case("step 1024", "step", 1024, (256, 32768, 4096), (1, 16), how="graph",
              rows="needed"),
        # a step whose logits come from a host-resident model: pinned inputs,
        # logits rows read in place over the host link
        _case("step 256 host-fed", "step", 256, (256, 32768, 4096), (1, 16), how="host",
              rows="needed"),
        # long reasoning traces: few requests, long contexts, 16-token spans
        # (128-row tiles) with the proposers' decode
        _case("attention long traces", "attn", 32, (8192, 32768), (16, 16), direction="S",
              decode_only=False),
        # student-verified ragged spans (2 to 32 rows per KV head) and GQA-8 decode
        _case("attention student verifies", "attn", 96, (256, 8192), (1, 16), direction="T",
              decode_only=False),
        # the proposal phase at a small batch: one decode token of 8 requests
        _case("decode 8", "attn", 8, (500, 16000), (1, 1), direction="half",
              decode_only=True),
        # a high-batch step with entropy takeover, by-products and the next
        # span's first token
        _case("score with rules 512", "score", 512, (2048, 4096), (4, 4), logits="zipf"),
        # the training direction: top-K lists, loss, dense bf16 logit gradient
        _case("loss and gradient 77", "train", 77, (1024, 8192), (1, 12), dense="bf16"),
        # full-vocabulary KL of a monitoring pass over an odd number of positions
        _case("full KL 333", "kl", 333, (1024, 8192), (1, 1)),
        # proposers' sampling: one row per request
        _case("sample 192", "sample", 192, (1024, 8192), (1, 1), logits="normal", sigma=3.0),
        # the step's K/V rows into both caches, one launch
        _case("append 64", "append", 64, (1024, 8192), (8, 8)),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "attn", "attn", "score", "train", "kl", "sample",
                       "append"])
    vocab = rng.choice([QWEN_VOCAB, QWEN_VOCAB, 8 * _log_int(rng, 512, 18992)])
    K = rng.choice([8, 16, 16, 16, 32])
    logits = rng.choice(["boost", "boost", "zipf", "normal"])
    direction = rng.choice(["S", "T", "half", "half"])
    hi = rng.choice([1, 4, 8, 16, 16, 24])
    span = (rng.choice([1, hi]), hi)
    R = _log_int(rng, 1, 768)
    top = _log_int(rng, 256, 32768)
    ctx = (max(span[1], rng.choice([top // 8, top // 3, 64])), top)
    if rng.random() < 0.3:
        ctx = (max(span[1], top // 32), top, max(span[1], top // 4))
    # no drawn case outgrows the listed full step (1024 requests, about 8,700
    # span positions and 6.8 M context tokens in each cache)
    most = int(6e6 / max(1.0, _mean_ctx({"ctx_lo": ctx[0], "ctx_hi": ctx[1],
                                         "ctx_median": ctx[2] if len(ctx) > 2 else 0})))
    R = max(1, min(R, most, 8000 // hi))
    kw = {"direction": direction, "vocab": vocab, "logits": logits, "K": K}
    if kind == "step":
        how = rng.choice(["calls", "graph", "graph", "host"])
        if how == "host":
            R = min(R, max(1, 3000 // hi))
        return _case("", "step", R, ctx, span, how=how,
                     rows="needed" if how == "host" else rng.choice(["all", "needed"]), **kw)
    if kind == "attn":
        return _case("", "attn", R, ctx, span, decode_only=rng.random() < 0.4, **kw)
    if kind == "score":
        return _case("", "score", R, ctx, span, **kw)
    if kind == "train":
        R = min(R, max(1, 3000 // hi))
        return _case("", "train", R, ctx, span, dense=rng.choice(["bf16", "f32", "none"]), **kw)
    if kind == "kl":
        return _case("", "kl", _log_int(rng, 8, 4000), (1024, 8192), (1, 1), **kw)
    if kind == "sample":
        return _case("", "sample", _log_int(rng, 1, 1024), (1024, 8192), (1, 1), vocab=vocab,
                     logits=rng.choice(["normal", "boost", "zipf"]),
                     sigma=rng.choice([1.0, 2.0, 3.0]))
    return _case("", "append", R, (ctx[0], min(ctx[1], 8192)) if ctx[0] <= 8192 else (4096, 8192),
                 span, **kw)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _quantiles(n):
    return (torch.arange(n, dtype=torch.float64) + 0.5) / n


def _ctx_of(case, u):
    lo, hi = case["ctx_lo"], case["ctx_hi"]
    if case["ctx_median"]:
        z = math.sqrt(2.0) * torch.erfinv((2 * u - 1).clamp(-1 + 1e-12, 1 - 1e-12))
        return torch.exp(math.log(case["ctx_median"]) + z).round().clamp(lo, hi).to(torch.int64)
    return (lo + torch.floor(u * (hi - lo + 1))).clamp(lo, hi).to(torch.int64)


def _mean_ctx(case):
    return float(_ctx_of(case, _quantiles(4096)).double().mean())


def _shapes(case, seed):
    """Lengths and drivers: the case's quantiles in an order of the seed's."""
    g = torch.Generator().manual_seed(seed)
    R = case["requests"]
    ctx = _ctx_of(case, _quantiles(R))[torch.randperm(R, generator=g)]
    lo, hi = case["span_lo"], case["span_hi"]
    span = (lo + torch.floor(_quantiles(R) * (hi - lo + 1))).clamp(lo, hi).to(torch.int64)
    if case["direction"] == "half":
        driver = (torch.arange(R) % 2).to(torch.uint8)
    else:
        driver = torch.full((R,), int(case["direction"] == "T"), dtype=torch.uint8)
    order = torch.randperm(R, generator=g)
    return ctx, span[order], driver[order], g


def _cu(lengths):
    out = torch.zeros(lengths.numel() + 1, dtype=torch.int32)
    out[1:] = torch.cumsum(lengths, 0)
    return out


def _page_table(ctx, g):
    n = (ctx + PAGE - 1) // PAGE
    total, R = int(n.sum()), ctx.numel()
    pt = torch.full((R, int(n.max())), -1, dtype=torch.int32)
    rows = torch.repeat_interleave(torch.arange(R), n)
    cols = torch.arange(total) - torch.repeat_interleave(torch.cumsum(n, 0) - n, n)
    pt[rows, cols] = torch.randperm(total, generator=g).to(torch.int32)
    return pt, total


def _normal(shape, gd):
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(generator=gd)


def _pools(hkv, pages, gd):
    return _normal((pages, hkv, PAGE, D), gd), _normal((pages, hkv, PAGE, D), gd)


def _logits(case, span, driver, gd):
    """Both models' rows and the proposed tokens (drawn from the proposer)."""
    V, T, R = case["vocab"], int(span.sum()), span.numel()
    req = torch.repeat_interleave(torch.arange(R), span).cuda()
    drv = driver.cuda()[req]
    out = [torch.empty((T, V), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    tokens = torch.empty(T, dtype=torch.int32, device="cuda")
    base = None
    if case["logits"] == "zipf":  # one rank permutation per request, both models share it
        base = torch.empty((R, V), dtype=torch.bfloat16, device="cuda")
        for r0 in range(0, R, 256):
            n = min(256, R - r0)
            rank = torch.rand((n, V), generator=gd, device="cuda").argsort(1)
            base[r0:r0 + n] = -1.1 * torch.log(rank.float() + 1.0)
    sigma = case.get("sigma", 3.0)
    for t0 in range(0, T, 512):
        t1 = min(T, t0 + 512)
        for x in out:
            y = torch.randn((t1 - t0, V), generator=gd, device="cuda")
            x[t0:t1] = y + base[req[t0:t1]] if base is not None else y * sigma
        s = drv[t0:t1] == 0
        e = torch.empty((t1 - t0, V), device="cuda").exponential_(generator=gd)
        prop = torch.where(s[:, None], out[0][t0:t1], out[1][t0:t1]).float()
        tok = (prop - torch.log(e)).argmax(1)
        tokens[t0:t1] = tok.to(torch.int32)
        if case["logits"] == "boost":
            rows = torch.arange(t0, t1, device="cuda")
            val = (8.1 + 8.0 * torch.rand(t1 - t0, generator=gd, device="cuda")).to(torch.bfloat16)
            out[1][rows, tok] = torch.where(s, val, out[1][rows, tok])
            out[0][rows, tok] = torch.where(s, out[0][rows, tok], val)
    return out[0], out[1], tokens


class State:
    pass


def prepare(case, seed):
    ctx, span, driver, g = _shapes(case, seed)
    gd = torch.Generator(device="cuda").manual_seed(seed + 7919)
    st = State()
    st.case, st.ctx, st.span, st.driver = case, ctx, span, driver
    {"step": _prep_step, "attn": _prep_attn, "score": _prep_score, "train": _prep_score,
     "kl": _prep_kl, "sample": _prep_sample, "append": _prep_append}[case["kind"]](st, g, gd)
    return st


def _prep_step(st, g, gd):
    c, ctx, span, driver = st.case, st.ctx, st.span, st.driver
    pt, ps = _page_table(ctx, g), _page_table(ctx, g)
    st.pt = {"t": pt[0], "s": ps[0]}
    tk, tv = _pools(HEADS["t"][1], pt[1], gd)
    sk, sv = _pools(HEADS["s"][1], ps[1], gd)
    ns, nt = int((driver == 0).sum()), int((driver == 1).sum())
    ls, lt, tokens = _logits(c, span, driver, gd)
    st.step = VerifyStep(tk, tv, sk, sv, ctx, span, driver, pt[0], ps[0],
                         _normal((int(span[driver == 0].sum()), HEADS["t"][0], D), gd),
                         _normal((int(span[driver == 1].sum()), HEADS["s"][0], D), gd),
                         _normal((ns, HEADS["s"][0], D), gd), _normal((nt, HEADS["t"][0], D), gd),
                         tokens, ls, lt, K=c["K"], rows=c["rows"])
    if c["how"] == "graph":
        st.graph = st.step.capture(overlap=True)
    elif c["how"] == "host":
        st.host, st.results = st.step.host_inputs(), st.step.host_results()
        st.graph = st.step.capture_from_host(st.host, st.results, host_logits=True)


def _batch(st, cache, which, q_len, idx, pt, gd):
    hq = HEADS[which][0]
    q = _normal((int(q_len.sum()), hq, D), gd)
    return ipd.AttnBatch(cache, q, _cu(q_len).cuda(), st.ctx[idx].to(torch.int32).cuda(),
                         pt[idx].contiguous().cuda(), torch.empty_like(q), int(q_len.max()),
                         int(st.ctx[idx].max()))


def _prep_attn(st, g, gd):
    st.verify, st.decode, st.parts = [], [], []
    for which in ("t", "s"):
        pt, pages = _page_table(st.ctx, g)
        cache = ipd.KVCache(*_pools(HEADS[which][1], pages, gd))
        ver = torch.nonzero(st.driver == (0 if which == "t" else 1)).flatten()
        prop = torch.nonzero(st.driver == (1 if which == "t" else 0)).flatten()
        if ver.numel() and not st.case["decode_only"]:
            b = _batch(st, cache, which, st.span[ver], ver, pt, gd)
            st.verify.append(b)
            st.parts.append((b, which, ver, st.span[ver], pt))
        if prop.numel():
            one = torch.ones(prop.numel(), dtype=torch.int64)
            b = _batch(st, cache, which, one, prop, pt, gd)
            st.decode.append(b)
            st.parts.append((b, which, prop, one, pt))
    st.ws = torch.empty(max(256, ipd.attn_workspace_size(st.verify, st.decode)), dtype=torch.uint8,
                        device="cuda")


def _prep_score(st, g, gd):
    c = st.case
    st.ls, st.lt, st.tokens = _logits(c, st.span, st.driver, gd)
    T, V, K, R = st.ls.shape[0], c["vocab"], c["K"], c["requests"]
    st.cu, st.drv = _cu(st.span).cuda(), st.driver.cuda()
    st.prefix = (st.ctx - st.span).to(torch.int32).cuda()
    st.out = ipd.alloc_score_outputs(R, T, "cuda")
    st.ws = torch.empty(max(256, ipd.score_workspace_size(R, T, V, K)), dtype=torch.uint8,
                        device="cuda")
    f = lambda: torch.empty(T, device="cuda")
    i = lambda *s: torch.empty(s, dtype=torch.int32, device="cuda")
    st.ent_s, st.ent_t, st.overlap = f(), f(), f()
    st.tks, st.tkt, st.next = i(T, K), i(T, K), i(R)
    if c["kind"] == "train":
        st.out8 = torch.zeros(8, device="cuda")
        st.gi, st.gv = i(T, 2 * K), torch.empty((T, 2 * K), device="cuda")
        dt = {"bf16": torch.bfloat16, "f32": torch.float32, "none": None}[c["dense"]]
        st.dense = None if dt is None else torch.empty((T, V), dtype=dt, device="cuda")


def _prep_kl(st, g, gd):
    st.ls, st.lt, _ = _logits(st.case, st.span, st.driver, gd)
    st.rev = torch.empty(st.ls.shape[0], device="cuda")
    st.fwd = torch.empty_like(st.rev)


def _prep_sample(st, g, gd):
    st.driver[:] = 0
    st.ls, st.lt, _ = _logits(st.case, st.span, st.driver, gd)
    n = st.ls.shape[0]
    st.rows = st.ls if st.case["logits"] != "boost" else st.lt
    st.draw = torch.randint(0, 1 << 40, (n,), generator=gd, device="cuda")
    st.tok = torch.empty(n, dtype=torch.int32, device="cuda")
    st.ws = torch.empty(max(8, ipd.sample_workspace_size(n, st.case["vocab"])), dtype=torch.uint8,
                        device="cuda")


def _prep_append(st, g, gd):
    st.appends, st.pools = [], []
    for which in ("t", "s"):
        pt, pages = _page_table(st.ctx, g)
        hkv = HEADS[which][1]
        # the pools hold what earlier steps wrote: zeros stand for it
        pool = [torch.zeros((pages, hkv, PAGE, D), dtype=torch.bfloat16, device="cuda")
                for _ in range(2)]
        st.pools += pool
        cache = ipd.KVCache(*pool)
        ver = torch.nonzero(st.driver == (0 if which == "t" else 1)).flatten()
        prop = torch.nonzero(st.driver == (1 if which == "t" else 0)).flatten()
        for idx, n in ((ver, st.span[ver]), (prop, torch.ones(prop.numel(), dtype=torch.int64))):
            if not idx.numel():
                continue
            total = int(n.sum())
            st.appends.append((cache, _normal((total, hkv, D), gd), _normal((total, hkv, D), gd),
                               _cu(n).cuda(), st.ctx[idx].to(torch.int32).cuda(),
                               pt[idx].contiguous().cuda()))


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(st):
    c = st.case
    kind = c["kind"]
    if kind == "step":
        if c["how"] == "calls":
            st.step.run()
        else:
            st.graph.replay()
        out = {"attn." + n: b.out for n, b, _, _ in st.step.batches}
        sc = dict(st.step.score)
        if c["rows"] == "needed":
            # a needed-rows pass defines these at the emitted positions only
            gone = sc["source"] == 255
            for n in TOKEN_OUTS:
                sc[n] = sc[n].masked_fill(gone, 0.0)
            del sc["covered"], sc["margin"]
        out.update(sc)
        out["out8"] = st.step.out8
        return out
    if kind == "attn":
        if c["decode_only"]:
            ipd.decode_attn(st.decode, SCALE, st.ws)
        else:
            ipd.verify_attn(st.verify, st.decode, SCALE, st.ws)
        return [b.out for b, _, _, _, _ in st.parts]
    if kind == "score":
        ipd.score_span_ex(st.ls, st.lt, st.tokens, st.cu, st.drv, st.prefix, c["K"], -1, st.out,
                          st.ws, ipd.RULE_ENTROPY_S, ipd.RULE_TOPK, TAU, 0.0, st.ent_s, st.ent_t,
                          st.overlap, st.tks, st.tkt, next_token=st.next, sample_seed=SAMPLE_SEED)
        return dict(st.out, entropy_s=st.ent_s, entropy_t=st.ent_t, overlap=st.overlap,
                    topk_s=st.tks, topk_t=st.tkt, next_token=st.next)
    if kind == "train":
        ipd.score_span_ex(st.ls, st.lt, st.tokens, st.cu, st.drv, st.prefix, c["K"], -1, st.out,
                          st.ws, topk_s=st.tks, topk_t=st.tkt)
        o = st.out
        ipd.split_loss(o["kl_rev"], o["kl_fwd"], o["source"], st.cu, o["n_emit"], None,
                       ipd.AGG_SEQ_MEAN_TOKEN_MEAN, ipd.DIR_SPLIT, st.out8)
        ipd.split_loss_grad(st.ls, st.lt, st.tks, st.tkt, o["source"], st.cu, o["n_emit"], None,
                            st.out8, c["K"], ipd.AGG_SEQ_MEAN_TOKEN_MEAN, ipd.DIR_SPLIT, 1.0,
                            st.gi, st.gv, st.dense)
        return dict(o, topk_s=st.tks, topk_t=st.tkt, out8=st.out8, grad_idx=st.gi, grad_val=st.gv,
                    **({} if st.dense is None else {"grad": st.dense}))
    if kind == "kl":
        ipd.full_kl(st.ls, st.lt, st.rev, st.fwd)
        return {"rev": st.rev, "fwd": st.fwd}
    if kind == "sample":
        ipd.sample(st.rows, SAMPLE_SEED, st.draw, st.tok, st.ws)
        return st.tok
    ipd.kv_append_many(st.appends)
    return st.pools


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _mean_span(case):
    return min((case["span_lo"] + case["span_hi"]) / 2.0, _mean_ctx(case))


def _needed_rows(case):
    """Expected logits rows a step needs: the verifier's up to the first
    transition, the proposer's at the emitted positions (about 0.61 of
    "boost" tokens are covered, of the others nearly all)."""
    p = 0.61 if case["logits"] == "boost" else 0.95
    lo, hi, total = case["span_lo"], case["span_hi"], 0.0
    share_t = {"S": 0.0, "T": 1.0, "half": 0.5}[case["direction"]]
    for k in range(lo, hi + 1):
        for stop, kept, share in ((1 - p, 0, 1 - share_t), (p, 1, share_t)):
            reach = sum((1 - stop) ** i for i in range(k))         # verifier rows
            emit = reach if kept else sum((1 - stop) ** (i + 1) for i in range(k))
            total += share * (reach + emit) / (hi - lo + 1)
    return case["requests"] * total


def _attn_work(case, verify=True):
    R, L, k = case["requests"], _mean_ctx(case), _mean_span(case)
    share = {"S": 1.0, "T": 0.0, "half": 0.5}[case["direction"]]  # student-driven requests
    byt = flo = 0.0
    for which, ver in (("t", share), ("s", 1.0 - share)):
        hq, hkv = HEADS[which]
        for n, rows in ((ver * R if verify else 0.0, k), ((1.0 - ver) * R, 1.0)):
            byt += n * (L * hkv * D * 2 * 2 + rows * hq * D * 2 * 2)
            flo += n * rows * hq * L * D * 4
    return byt, flo


def work(case):
    V, R = case["vocab"], case["requests"]
    T = R * _mean_span(case)
    kind = case["kind"]
    if kind == "step":
        byt, flo = _attn_work(case)
        rows = 2 * T if case["rows"] == "all" else min(2 * T, _needed_rows(case))
        return {"bytes": byt + rows * V * 2 + T * 26 + R * 14, "flops": flo + rows * V * 4}
    if kind == "attn":
        byt, flo = _attn_work(case, not case["decode_only"])
        return {"bytes": byt, "flops": flo}
    if kind == "score":
        return {"bytes": (2 * T + R) * V * 2 + T * (42 + 8 * case["K"]), "flops": 2 * T * V * 6 + R * V * 20}
    if kind == "train":
        dense = {"bf16": 2, "f32": 4, "none": 0}[case["dense"]]
        return {"bytes": 2 * T * V * 2 + T * V * dense + T * (26 + 24 * case["K"]), "flops": 2 * T * V * 4}
    if kind == "kl":
        return {"bytes": 2 * R * V * 2 + 8 * R, "flops": R * V * 14}
    if kind == "sample":
        return {"bytes": R * V * 2 + 12 * R, "flops": R * V * 20}
    share = {"S": 1.0, "T": 0.0, "half": 0.5}[case["direction"]]
    rows = [share * T + (1 - share) * R, (1 - share) * T + share * R]
    return {"bytes": sum(n * HEADS[w][1] * D * 2 * 2 * 2 for n, w in zip(rows, ("t", "s"))), "flops": 0}


def tolerance(case):
    kind = case["kind"]
    if kind in ("sample", "append"):
        return "exact"  # token ids of a bit-exact draw, copied bytes
    if kind in ("step", "attn"):
        # bf16 attention outputs: two fp32-accurate results round apart by a
        # bf16 step (2^-8 of a value) at a few per cent of the values
        return {"rel": 4e-3, "max": 0.03}
    if kind == "score":
        # fp32 sums; an entropy within 1e-5 of the threshold may decide either way
        return {"rel": 1e-5, "max": 1e-3, "differ": 5e-3}
    if kind == "train":
        return {"rel": 4e-3 if case["dense"] == "bf16" else 1e-5, "max": 0.02}
    return {"rel": 1e-5, "max": 1e-3}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------
def _exact_attn(batch, q_len, ctx, pt, which):
    hq, hkv = HEADS[which]
    G = hq // hkv
    q, out = batch._keep[0], torch.empty(batch.out.shape, dtype=torch.float64, device="cuda")
    kp, vp = batch.cache.k_pages, batch.cache.v_pages
    t = 0
    for r in range(q_len.numel()):
        n, L = int(q_len[r]), int(ctx[r])
        pages = pt[r, :(L + PAGE - 1) // PAGE].to("cuda", torch.int64)
        K, V = (p[pages].transpose(0, 1).reshape(hkv, -1, D)[:, :L].double() for p in (kp, vp))
        Q = q[t:t + n].double().view(n, hkv, G, D).permute(1, 0, 2, 3).reshape(hkv, n * G, D)
        S = (Q @ K.transpose(1, 2)) * SCALE
        lim = torch.arange(L - n, L, device="cuda").repeat_interleave(G)
        S.masked_fill_(torch.arange(L, device="cuda")[None, None, :] > lim[None, :, None], -math.inf)
        O = torch.softmax(S, 2) @ V
        out[t:t + n] = O.view(hkv, n, G, D).permute(1, 0, 2, 3).reshape(n, hq, D)
        t += n
    return out


def _topk(rows, K):
    """Token ids of the K largest logits, ties to the smaller id."""
    b = rows.view(torch.int16).to(torch.int64) & 0xFFFF
    b = torch.where(b == 0x8000, torch.zeros_like(b), b)
    o = torch.where(b >= 0x8000, 0xFFFF - b, b + 0x8000)
    ids = torch.arange(rows.shape[1], device=rows.device)
    return torch.topk((o << 32) + (0x7FFFFFFF - ids), K, dim=1).indices


def _exact_score(st, ls, lt, tokens, K, rules=False):
    """Per-position values of a vocabulary pass, the verdict, and the loss."""
    T = tokens.numel()
    f = {n: torch.empty(T, dtype=torch.float64, device="cuda")
         for n in TOKEN_OUTS + ("margin", "entropy_s", "entropy_t", "overlap")}
    ids = [torch.empty((T, K), dtype=torch.int64, device="cuda") for _ in range(2)]
    cov_k = torch.empty(T, dtype=torch.bool, device="cuda")
    drv = torch.repeat_interleave(st.driver, st.span).cuda()
    for t0 in range(0, T, 128):
        t1 = min(T, t0 + 128)
        rows = torch.arange(t1 - t0, device="cuda")
        x = tokens[t0:t1].long()
        lx, lz, en, tk = [], [], [], []
        for m, src in enumerate((ls, lt)):
            l = src[t0:t1].double()
            z = torch.logsumexp(l, 1)
            lz.append(z)
            en.append(z - (torch.exp(l - z[:, None]) * l).sum(1))
            lx.append(l[rows, x])
            tk.append(_topk(src[t0:t1], K))
            ids[m][t0:t1] = tk[m]
        f["logp_s"][t0:t1], f["logp_t"][t0:t1] = lx[0] - lz[0], lx[1] - lz[1]
        f["feedback"][t0:t1] = (lx[1] - lz[1]) - (lx[0] - lz[0])
        f["entropy_s"][t0:t1], f["entropy_t"][t0:t1] = en
        dup = (tk[1][:, :, None] == tk[0][:, None, :]).any(2)
        f["overlap"][t0:t1] = dup.double().mean(1)
        sup = torch.cat(tk, 1)
        gone = torch.cat([torch.zeros_like(dup), dup], 1)
        lp = []
        for src in (ls, lt):
            a = src[t0:t1].gather(1, sup).double().masked_fill(gone, -math.inf)
            lp.append(torch.log_softmax(a, 1))
        for n, a, b in (("kl_rev", lp[0], lp[1]), ("kl_fwd", lp[1], lp[0])):
            term = torch.where(gone, torch.zeros_like(a), torch.exp(a) * (a - b))
            f[n][t0:t1] = term.sum(1)
        d = drv[t0:t1] == 0
        ver = torch.where(d[:, None], tk[1], tk[0])
        cov_k[t0:t1] = (ver == x[:, None]).any(1)
        kth = torch.where(d, lt[t0:t1].gather(1, tk[1][:, -1:])[:, 0].double(),
                          ls[t0:t1].gather(1, tk[0][:, -1:])[:, 0].double())
        f["margin"][t0:t1] = torch.where(d, lx[1], lx[0]) - kth
    cov = cov_k
    if rules:  # entropy takeover, top-K handback
        cov = torch.where(drv == 0, f["entropy_s"] <= TAU, cov_k)
        f["margin"] = torch.where(drv == 0, TAU - f["entropy_s"], f["margin"])
    source = torch.full((T,), 255, dtype=torch.int64)
    c, t, n_emit = cov.cpu().tolist(), 0, []
    for k, d in zip(st.span.tolist(), st.driver.tolist()):
        n = 0
        for i in range(k):
            if d == 0 and not c[t + i]:
                break
            n = i + 1
            if d == 1 and c[t + i]:
                break
        source[t:t + n] = d
        n_emit.append(n)
        t += k
    f["source"], f["n_emit"], f["ids"] = source.cuda(), torch.tensor(n_emit), ids
    w = torch.where(f["source"] == 0, f["kl_rev"],
                    torch.where(f["source"] == 1, f["kl_fwd"], torch.zeros_like(f["kl_rev"])))
    req = torch.repeat_interleave(torch.arange(st.span.numel()), st.span).cuda()
    per = torch.zeros(st.span.numel(), dtype=torch.float64, device="cuda").index_add_(0, req, w)
    ne = f["n_emit"].cuda().double()
    numer, denom = (per[ne > 0] / ne[ne > 0]).sum(), (ne > 0).double().sum()
    n_on, n_off = (f["source"] == 0).double().sum(), (f["source"] == 1).double().sum()
    zero = torch.zeros((), dtype=torch.float64, device="cuda")
    f["out8"] = torch.stack([numer / denom if denom > 0 else zero, w[f["source"] == 0].sum(),
                             w[f["source"] == 1].sum(), n_on, n_off,
                             n_off / (n_on + n_off) if n_on + n_off > 0 else zero, numer, denom])
    f["req"], f["denom"] = req, denom
    return f


def _exact_grad(st, f, K):
    T, V = st.ls.shape
    sup = torch.cat(f["ids"], 1)
    dup = (f["ids"][1][:, :, None] == f["ids"][0][:, None, :]).any(2)
    gone = torch.cat([torch.zeros_like(dup), dup], 1)
    a = torch.log_softmax(st.ls.gather(1, sup).double().masked_fill(gone, -math.inf), 1)
    b = torch.log_softmax(st.lt.gather(1, sup).double().masked_fill(gone, -math.inf), 1)
    diff = torch.where(gone, torch.zeros_like(a), a - b)
    rev = torch.exp(a) * (diff - f["kl_rev"][:, None])
    fwd = torch.exp(a) - torch.exp(b)
    w = 1.0 / (f["denom"] * f["n_emit"].cuda().double()[f["req"]])
    src = f["source"][:, None]
    v = torch.where(src == 0, rev, fwd) * w[:, None]
    v = torch.where((src == 255) | gone, torch.zeros_like(v), v)
    if st.case["dense"] == "none":
        return v, None
    dense = torch.zeros((T, V), dtype=torch.float64 if T * V < 2e9 else torch.float32,
                        device="cuda")
    return v, dense.scatter_add_(1, sup, v.to(dense.dtype))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("sample", "append"):
        return None  # whole values and copied bytes: compared exactly
    st = prepare({**case, "how": "calls"} if kind == "step" else case, seed)
    if kind == "attn":
        return [_exact_attn(b, n, st.ctx[idx], pt[idx], w) for b, w, idx, n, pt in st.parts]
    if kind == "kl":
        rev, fwd = [], []
        for t in range(0, st.ls.shape[0], 128):
            a, b = (torch.log_softmax(x[t:t + 128].double(), 1) for x in (st.ls, st.lt))
            rev.append((torch.exp(a) * (a - b)).sum(1))
            fwd.append((torch.exp(b) * (b - a)).sum(1))
        return {"rev": torch.cat(rev), "fwd": torch.cat(fwd)}
    if kind == "step":
        s = st.step
        out = {}
        for n, b, idx, cname in s.batches:
            which = cname[0]
            q_len = st.span[idx] if n.startswith("verify") else torch.ones_like(st.span[idx])
            out["attn." + n] = _exact_attn(b, q_len, st.ctx[idx], st.pt[which][idx], which)
        f = _exact_score(st, s.logits_s, s.logits_t, s.tokens, case["K"])
        gone = f["source"] == 255
        for n in TOKEN_OUTS:
            out[n] = f[n].masked_fill(gone, 0.0) if case["rows"] == "needed" else f[n]
        if case["rows"] == "all":
            out["margin"] = f["margin"]
        out["out8"] = f["out8"]
        return out
    f = _exact_score(st, st.ls, st.lt, st.tokens, case["K"], rules=kind == "score")
    out = {n: f[n] for n in TOKEN_OUTS + ("margin",)}
    if kind == "score":
        out.update({n: f[n] for n in ("entropy_s", "entropy_t", "overlap")})
        return out
    out["out8"] = f["out8"]
    out["grad_val"], dense = _exact_grad(st, f, case["K"])
    if dense is not None:
        out["grad"] = dense
    return out
