"""Measured work of the PCED decode-step library: its public entry points over
the sizes that programs run them at.

Four kinds of case:

* ``attn``   ``decode_attention``: one layer of decode attention, every
  sequence over its own cache (a program with its own layers calls it once per
  layer and step);
* ``lm_head`` ``lm_head_logprobs``: the log-probabilities of every expert;
* ``score``  ``relevance`` + ``adacad_beta`` + ``contrastive_select``: the
  first token of a decode from log-probabilities the program holds;
* ``step``   ``Decoder.step``: the whole decode step, the call a serving loop
  makes for every token.  A pass is the first step of a request: the lengths and
  the step counter go back to where the request began, then one step.

Shapes are those of the synthetic workloads (``synth``) and of the tests; the
inputs are generated here, from the seed alone.
"""
import math

import numpy as np
import torch

import paper_2601_08670_gb300 as pced

GAMMA = 2.5
RMS_EPS = 1e-6
BETA0 = 0.5
QUERY = 32     # rows of the question, which every cache holds after its document
ROOM = 64      # rows kept free in every cache for the tokens to come

HEADS = {  # name: (query heads, kv heads, head dim)
    "8/2/64": (8, 2, 64),        # the tiny workload
    "16/2/64": (16, 2, 64),      # eight query heads per kv head
    "32/8/128": (32, 8, 128),    # Llama-3-8B shapes
    "28/4/128": (28, 4, 128),    # Qwen2-7B shapes
}


# ------------------------------------------------------------------- the cases
def listed():
    return [
        # the tiny workload's layer: the smallest call, where launches count
        dict(name="attn_tiny", kind="attn", heads="8/2/64", B=1, N=2, docs="fixed", lo=257, hi=257, query=0),
        # one layer of a Llama-3-8B-shaped decode over eight documents of 2048 rows
        dict(name="attn_docs", kind="attn", heads="32/8/128", B=1, N=8, docs="fixed", lo=2049, hi=2049, query=QUERY),
        # one layer of a Qwen2-7B-shaped decode: seven query heads per kv head, longer documents
        dict(name="attn_gqa7", kind="attn", heads="28/4/128", B=1, N=16, docs="fixed", lo=4097, hi=4097, query=QUERY),
        # sixteen queries at once, ragged documents around 1024 rows: the largest layer
        dict(name="attn_batch", kind="attn", heads="32/8/128", B=16, N=16, docs="normal", lo=256, hi=2048,
             query=QUERY),
        # the vocabulary scores of one query's experts
        dict(name="lm_head_docs", kind="lm_head", S=9, d=4096, V=128256),
        # ... and of sixteen queries' experts at once
        dict(name="lm_head_batch", kind="lm_head", S=272, d=4096, V=128256),
        # first token from materialised log-probabilities: relevance, beta, choice
        dict(name="score_docs", kind="score", B=1, N=8, V=128256),
        # the tiny workload's whole step: launch latency
        step_case("step_tiny", "8/2/64", B=1, N=2, L=1, V=8192, docs="fixed", lo=256, hi=256, query=0),
        # the headline workload: Llama-3-8B shapes, eight documents of 2048 rows,
        # replayed as a CUDA graph as a serving loop does
        step_case("step_docs", "32/8/128", B=1, N=8, L=32, V=128256, docs="fixed", lo=2048, hi=2048, graph=True),
        # thirty-two ragged documents, rotary positions
        step_case("step_ragged", "32/8/128", B=1, N=32, L=32, V=128256, docs="uniform", lo=512, hi=8192, rope=5e5),
        # sixteen queries over paged caches: the largest step
        step_case("step_batch", "32/8/128", B=16, N=16, L=32, V=128256, docs="normal", lo=256, hi=2048, paged=256),
        # the experts mixed in probability space instead of Eq. 3's maximum, four layers
        step_case("step_moe", "32/8/128", B=1, N=8, L=4, V=128256, docs="fixed", lo=2048, hi=2048, agg=pced.AGG_MOE),
    ]


def step_case(name, heads, B, N, L, V, docs, lo, hi, query=QUERY, paged=0, rope=0.0, agg=0, logit=False, first=False,
              graph=False):
    c = dict(kind="step", heads=heads, B=B, N=N, L=L, V=V, docs=docs, lo=lo, hi=hi, query=query, paged=paged,
             rope=float(rope), agg=agg, logit=logit, first=first, graph=graph)
    return dict(c, name=name) if name else c


def _log(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_docs(rng, rows):
    """Document lengths: about `rows` each."""
    how = rng.choice(["fixed", "uniform", "normal"])
    if how == "fixed":
        return how, rows, rows
    return how, max(1, rows // rng.randint(2, 16)), rows


def _draw_batch(rng):
    """(queries, experts per query) with at most 272 sequences."""
    B = rng.choice([1, 1, 1, 2, 3, 5, 8, 16])
    return B, _log(rng, 1, min(64, 272 // B - 1))


def draw(rng):
    kind = rng.choice(["attn", "attn", "lm_head", "score", "step", "step"])
    if kind == "lm_head":
        d = rng.choice([512, 1024, 1792, 3584, 4096])
        return dict(kind=kind, S=_log(rng, 1, 272), d=d, V=_log(rng, 1000, 151936))
    B, N = _draw_batch(rng)
    if kind == "score":
        return dict(kind=kind, B=B, N=N, V=_log(rng, 1000, 151936))
    heads = rng.choice(sorted(HEADS))
    S = B * (N + 1)
    # rows a layer: at most about what the largest listed cases hold
    how, lo, hi = _draw_docs(rng, _log(rng, 16, max(32, min(8192, 270_000 // S))))
    if kind == "attn":
        return dict(kind=kind, heads=heads, B=B, N=N, docs=how, lo=lo, hi=hi, query=QUERY)
    agg = rng.choice([pced.AGG_MAX, pced.AGG_MAX, pced.AGG_MAX, pced.AGG_MOE, pced.AGG_POE])
    return step_case(None, heads, B=B, N=N, L=_log(rng, 1, 28), V=_log(rng, 1000, 151936), docs=how, lo=lo, hi=hi,
                     paged=rng.choice([0, 0, 64, 192, 256]), rope=rng.choice([0.0, 1e4, 5e5]), agg=agg,
                     logit=agg == pced.AGG_MAX and rng.random() < 0.25, first=rng.random() < 0.2,
                     graph=rng.random() < 0.5)


# ----------------------------------------------------------------- the inputs
def _lengths(c):
    """Live rows of every sequence, query-major, amateur first (a property of the case, not of the seed)."""
    rng = np.random.default_rng([c["B"], c["N"], c["lo"], c["hi"]])
    n, lo, hi = c["B"] * c["N"], c["lo"], c["hi"]
    if c["docs"] == "fixed":
        docs = np.full(n, lo)
    elif c["docs"] == "uniform":
        docs = rng.integers(lo, hi, endpoint=True, size=n)
    else:
        docs = np.clip(np.rint(rng.normal((lo + hi) / 2, max(1.0, (hi - lo) / 7), size=n)), lo, hi)
    out = np.empty((c["B"], c["N"] + 1), np.int64)
    out[:, 0] = QUERY + (1 if c["kind"] == "attn" else 0)
    out[:, 1:] = docs.reshape(c["B"], c["N"]) + c["query"]
    return out.reshape(-1)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(shape, sigma, g, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, sigma, generator=g)


def _dev(a, dtype):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def _slabs(lens, Hkv, D):
    cap = lens + ROOM
    sizes = Hkv * cap * D
    off = np.concatenate([[0], np.cumsum(sizes)[:-1]])
    return cap, off, int(sizes.sum())


def _pages(lens, P, seed):
    """Block table in which the blocks lie scattered over the pool, as a serving allocator leaves them."""
    cap = lens + ROOM
    nblk = (cap + P - 1) // P
    order = np.random.default_rng(seed).permutation(int(nblk.sum()))
    table = np.full((len(cap), int(nblk.max())), -1, np.int64)
    at = 0
    for s, n in enumerate(nblk):
        table[s, :n] = order[at:at + n]
        at += n
    return cap, table, int(nblk.sum())


def prepare(case, seed):
    return {"attn": _prepare_attn, "lm_head": _prepare_lm_head, "score": _prepare_score,
            "step": _prepare_step}[case["kind"]](case, seed)


def _prepare_attn(c, seed):
    Hq, Hkv, D = HEADS[c["heads"]]
    g, lens = _gen(seed), _lengths(c)
    S = len(lens)
    cap, off, elems = _slabs(lens, Hkv, D)
    st = dict(case=c, q=_normal((S, Hq, D), 1.0, g), k=_normal(elems, 1.0, g), v=_normal(elems, 1.0, g),
              off=_dev(off, torch.int64), cap=_dev(cap, torch.int32), lens=_dev(lens, torch.int32), Hkv=Hkv,
              total_cap=int(cap.sum()), host=(lens, cap, off))
    st["out"] = torch.empty((S, Hq, D), dtype=torch.float32, device="cuda")
    st["ws"] = pced.workspace(pced.decode_attention_workspace_size(S, Hq, Hkv, D), "cuda")
    return st


def _prepare_lm_head(c, seed):
    g, S, d, V = _gen(seed), c["S"], c["d"], c["V"]
    return dict(case=c, h=_normal((S, d), 1.0, g), w=_normal((V, d), 0.02, g),
                lp=torch.empty((S, V), dtype=torch.float32, device="cuda"),
                lse=torch.empty(S, dtype=torch.float32, device="cuda"),
                ws=pced.workspace(pced.lm_head_workspace_size(S, V), "cuda"))


def _prepare_score(c, seed):
    g, B, N, V = _gen(seed), c["B"], c["N"], c["V"]
    z0 = _normal((B, 1, V), 2.5, g, torch.float32)
    z = _normal((B, N + 1, V), 1.5, g, torch.float32)
    z[:, :1] = 0.0
    z += z0  # the experts agree with the amateur in part
    lp = torch.log_softmax(z.view(B * (N + 1), V), dim=1)
    ws = max(int(pced.lib().pced_adacad_beta_workspace_size(B, N, V)), pced.contrastive_select_workspace_size(B, N, V))
    return dict(case=c, lp=lp, ret=torch.empty((B, N), device="cuda").uniform_(-1.0, 1.0, generator=g),
                rer=_normal((B, N), 2.0, g, torch.float32), ws=pced.workspace(ws, "cuda"))


def _prepare_step(c, seed):
    Hq, Hkv, D = HEADS[c["heads"]]
    B, N, L, V, P, d = c["B"], c["N"], c["L"], c["V"], c["paged"], Hq * D
    g, lens = _gen(seed), _lengths(c)
    S = len(lens)
    table = None
    if P:
        cap, table, nblocks = _pages(lens, P, seed)
        off, layer = np.zeros(S, np.int64), nblocks * Hkv * P * D
    else:
        cap, off, layer = _slabs(lens, Hkv, D)
    kv = _normal((2, L * layer), 1.0, g)
    embed, w = _normal((V, d), 1.0, g), _normal((V, d), 0.02, g)
    base = _dev(lens, torch.int32)
    br = torch.empty((2, B, N), device="cuda")
    br[0] = BETA0
    br[1].uniform_(0.0, 1.0, generator=g)
    dec = pced.Decoder(pced.dims(B, N, L, Hq, Hkv, D, V), embed=embed, w_unembed=w, k_cache=kv[0], v_cache=kv[1],
                       layer_elems=layer, kv_offset=_dev(off, torch.int64), cap=_dev(cap, torch.int32),
                       seq_len=base.clone(), beta=br[0], r=br[1], gamma=GAMMA, max_steps=ROOM,
                       total_cap=int(cap.sum()), rms_eps=RMS_EPS, keep_hidden=True, dynamic_beta=c["first"],
                       block_table=None if table is None else _dev(table, torch.int32), block_rows=P,
                       rope_theta=c["rope"], score_mode=pced.SCORE_LOGIT if c["logit"] else pced.SCORE_LOGPROB,
                       aggregation=c["agg"])
    st = dict(case=c, dec=dec, base=base, kv=kv, embed=embed, w=w, br=br, lens=lens, cap=cap, off=off, layer=layer,
              table=table)
    # where the K and V row of the new token goes, in every layer and kv-head:
    # a view for each sequence, or, past what can be returned one by one, the rows' numbers
    if S <= 33:
        st["rows"] = [torch.as_strided(kv, (2, L, Hkv, D), (L * layer, layer, (P or int(cap[s])) * D, 1), at)
                      for s, at in enumerate(_row_offsets(st, Hkv, D))]
    else:
        l, h, t = np.arange(L)[:, None, None], np.arange(Hkv)[None, None, :], np.arange(2)[:, None, None, None]
        step = np.asarray([P or int(n) for n in cap])[None, :, None]
        rows = (np.asarray(_row_offsets(st, Hkv, D))[None, :, None] + l * layer) // D + h * step
        st["row_ids"] = _dev((rows[None] + t * (L * layer // D)).reshape(-1), torch.int64)
    if c["graph"]:
        _one_step(st)  # what a program does before it captures
        torch.cuda.synchronize()
        gr = torch.cuda.CUDAGraph()
        with torch.cuda.graph(gr):
            _one_step(st)
        st["graph"] = gr
    return st


def _row_offsets(st, Hkv, D):
    """Element of kv-head 0's new row of every sequence, in layer 0 of the K cache."""
    out, P = [], st["case"]["paged"]
    for s, n in enumerate(st["lens"]):
        n = int(n)
        out.append(int(st["table"][s, n // P]) * Hkv * P * D + (n % P) * D if P else int(st["off"][s]) + n * D)
    return out


# ------------------------------------------------------------------- one pass
def _one_step(st):
    dec = st["dec"]
    dec.seq_len.copy_(st["base"])  # the request's caches as they were loaded
    dec.step_t.zero_()
    if st["case"]["first"]:
        dec.args.beta_from_step = 1  # as a new Decoder(dynamic_beta=True) has it
    dec.step()


def run(st):
    c = st["case"]
    if c["kind"] == "attn":
        return pced.decode_attention(st["q"], st["k"], st["v"], st["off"], st["cap"], st["lens"], st["Hkv"],
                                     st["total_cap"], out=st["out"], ws=st["ws"])
    if c["kind"] == "lm_head":
        lp, lse = pced.lm_head_logprobs(st["h"], st["w"], logprobs=st["lp"], lse=st["lse"], ws=st["ws"])
        return dict(logprobs=lp, lse=lse)
    if c["kind"] == "score":
        r = pced.relevance(st["ret"], pced.RET_DENSE, st["rer"])
        beta = pced.adacad_beta(st["lp"], c["B"], c["N"], ws=st["ws"])
        token, expert, score = pced.contrastive_select(st["lp"], beta, r, GAMMA, ws=st["ws"])
        return dict(r=r, beta=beta, token=token, expert=expert, score=score)
    if c["graph"]:
        st["graph"].replay()
    else:
        _one_step(st)
    dec = st["dec"]
    out = dict(hidden=dec.hidden, lse=dec.lse, score=dec.score_out, seq_len=dec.seq_len, step=dec.step_t)
    if c["B"] == 1:
        # the choice itself; of several queries one may be so near a tie that
        # another order of sums in 16-bit layers turns it: there the score says which it was
        out.update(token=dec.token_out, expert=dec.expert_out)
    if c["first"]:
        out["beta"] = dec.beta
    Hq, Hkv, D = HEADS[c["heads"]]
    out["rows"] = (st["rows"] if "rows" in st else
                   st["kv"].view(-1, D).index_select(0, st["row_ids"]).view(2, c["L"], -1, Hkv, D))
    return out


# ------------------------------------------------------------ what it has to do
def work(case):
    if case["kind"] == "lm_head":
        S, d, V = case["S"], case["d"], case["V"]
        return {"bytes": 2 * (V * d + S * d) + 4 * (S * V + S), "flops": 2 * S * V * d}
    B, N = case["B"], case["N"]
    S = B * (N + 1)
    if case["kind"] == "score":
        return {"bytes": 4 * S * case["V"] + 24 * B * N, "flops": 30 * B * N * case["V"]}
    Hq, Hkv, D = HEADS[case["heads"]]
    lens = _lengths(case)
    if case["kind"] == "attn":
        rows = int(lens.sum())
        return {"bytes": rows * 4 * Hkv * D + 6 * S * Hq * D, "flops": 4 * rows * Hq * D}
    d, L, V = Hq * D, case["L"], case["V"]
    rows = int((lens + 1).sum())
    return {"bytes": L * rows * 4 * Hkv * D + 2 * V * d + 2 * B * d + 2 * S * d + 4 * S,
            "flops": L * 4 * rows * d + 2 * S * V * d}


def tolerance(case):
    # about four times the largest error against `exact` that was measured
    if case["kind"] == "attn":
        return {"rel": 8e-6}  # fp32 scores and sums of bf16 inputs, probabilities held to 16 bits or more: 1.9e-6
    if case["kind"] == "lm_head":
        return {"rel": 3e-6}  # fp32 sums of exact bf16 products: 7e-7
    if case["kind"] == "score":
        return {"rel": 4e-7}  # fp32 terms, sums in 64 bits: 8e-8
    # every layer's queries, the appended rows and the final hidden state are rounded
    # to bf16: a last-bit difference of an fp32 sum turns a few of them (by up to 2^-7
    # of a value) and travels through the layers: 7.3e-4
    return {"rel": 3e-3, "max": 3e-2}


# --------------------------------------------------------- the same in 64 bits
def exact(case, seed):
    with torch.no_grad():
        return {"attn": _exact_attn, "lm_head": _exact_lm_head, "score": _exact_score,
                "step": _exact_step}[case["kind"]](case, seed)


def _attend(q, k, v):
    """softmax(q k^T / sqrt(D)) v of one sequence: q [Hkv, G, D], k and v [Hkv, n, D], fp64."""
    return torch.softmax(q @ k.transpose(1, 2) / math.sqrt(q.shape[-1]), dim=2) @ v


def _exact_attn(c, seed):
    st = _prepare_attn(c, seed)
    Hq, Hkv, D = HEADS[c["heads"]]
    lens, cap, off = st["host"]
    out = torch.empty((len(lens), Hq, D), dtype=torch.float64, device="cuda")
    for s, n in enumerate(lens):
        part = slice(int(off[s]), int(off[s] + Hkv * cap[s] * D))
        k, v = (st[x][part].view(Hkv, -1, D)[:, :n].double() for x in "kv")
        out[s] = _attend(st["q"][s].double().view(Hkv, -1, D), k, v).reshape(Hq, D)
    return out


def _logits(h, w):
    return torch.cat([h.double() @ p.double().T for p in w.split(16384)], dim=1)


def _exact_lm_head(c, seed):
    st = _prepare_lm_head(c, seed)
    z = _logits(st["h"], st["w"])
    lse = torch.logsumexp(z, dim=1)
    return dict(logprobs=z.sub_(lse[:, None]), lse=lse)


def _jsd_bits(lp):
    """Jensen-Shannon divergence of each expert from its amateur: lp [B, N + 1, V] -> [B, N]."""
    a, k = lp[:, :1], lp[:, 1:]
    m = torch.logaddexp(a, k) - math.log(2.0)
    return 0.5 * (k.exp() * (k - m) + a.exp() * (a - m)).sum(2) / math.log(2.0)


def _choose(lp, beta, bias):
    """(token, expert, score) of Eq. 2 and Eq. 3: lp [B, N + 1, V], beta and bias [B, N]."""
    s = (1 + beta[:, :, None]) * lp[:, 1:] - beta[:, :, None] * lp[:, :1] + bias[:, :, None]
    best, expert = s.max(dim=1)
    score, token = best.max(dim=1)
    return token.int(), expert.gather(1, token[:, None])[:, 0].int() + 1, score


def _exact_score(c, seed):
    st = _prepare_score(c, seed)
    B, N, V, eps = c["B"], c["N"], c["V"], 1e-8
    a = ((st["ret"].double() + 1) / 2).clamp(0, 1 - eps)
    b = torch.sigmoid(st["rer"].double()).clamp(0, 1 - eps)
    r = 2 * a * b / (a + b + eps)
    lp = st["lp"].double().view(B, N + 1, V)
    beta = _jsd_bits(lp)
    token, expert, score = _choose(lp, beta, GAMMA * r.clamp(1e-8, 1.0).log())
    return dict(r=r, beta=beta, token=token, expert=expert, score=score)


def _rope(u, pos, theta):
    """Rotate-half embedding of u [S, H, D] at positions pos [S] (frequencies and angles in fp32)."""
    D = u.shape[2]
    f = (theta ** (-2.0 * np.arange(D // 2) / D)).astype(np.float32)
    ang = _dev(np.asarray(pos, np.float32)[:, None] * f[None], torch.float32).double()[:, None]
    a, b = u[..., :D // 2], u[..., D // 2:]
    return torch.cat([a * ang.cos() - b * ang.sin(), b * ang.cos() + a * ang.sin()], dim=2)


def _exact_step(c, seed):
    st = _prepare_step(dict(c, graph=False), seed)
    Hq, Hkv, D = HEADS[c["heads"]]
    B, N, L, P, S, d, layer = c["B"], c["N"], c["L"], c["paged"], len(st["lens"]), Hq * D, st["layer"]
    rows = torch.empty((2, L, S, Hkv, D), dtype=torch.float64, device="cuda")
    table = _dev(st["table"], torch.int64) if P else None

    def cached(part, l, s, n):
        mem = st["kv"][part, l * layer:(l + 1) * layer]
        if P:
            return mem.view(-1, Hkv, P, D)[table[s, :(n + P - 1) // P]].transpose(0, 1).reshape(Hkv, -1, D)[:, :n]
        at = int(st["off"][s])
        return mem[at:at + Hkv * int(st["cap"][s]) * D].view(Hkv, -1, D)[:, :n]

    def rounded(x):  # bf16(rmsnorm(x)), and u itself
        u = x / torch.sqrt((x * x).mean(1, keepdim=True) + RMS_EPS)
        return u, u.bfloat16().double()

    x = st["embed"][0].double().expand(S, d).clone()  # the first token follows token 0
    for l in range(L):
        u, ub = rounded(x)
        q, k, v = ub.view(S, Hq, D), ub.view(S, Hq, D)[:, :Hkv], ub.view(S, Hq, D)[:, Hkv:2 * Hkv]
        if c["rope"]:
            ur = _rope(u.view(S, Hq, D), st["lens"], c["rope"]).bfloat16().double()
            q, k = ur, ur[:, :Hkv]
        rows[0, l], rows[1, l] = k, v
        o = torch.empty_like(x)
        for s, n in enumerate(st["lens"]):
            ks, vs = (torch.cat([cached(i, l, s, int(n)).double(), rows[i, l, s][:, None]], dim=1) for i in (0, 1))
            o[s] = _attend(q[s].view(Hkv, -1, D), ks, vs).reshape(-1)
        x = x + o
    h = rounded(x)[1]
    z = _logits(h, st["w"])
    lse = torch.logsumexp(z, dim=1)
    lp = (z - lse[:, None]).view(B, N + 1, -1)
    r = st["br"][1].double().clamp(1e-8, 1.0)
    beta = _jsd_bits(lp) if c["first"] else torch.full_like(r, BETA0)
    if c["agg"] == pced.AGG_MAX:
        token, expert, score = _choose(z.view(B, N + 1, -1) if c["logit"] else lp, beta, GAMMA * r.log())
    else:
        p = torch.log_softmax((1 + beta[:, :, None]) * lp[:, 1:] - beta[:, :, None] * lp[:, :1], dim=2)
        lw = (r / r.sum(1, keepdim=True)).log()[:, :, None]
        mixed = torch.logsumexp(lw + p, dim=1) if c["agg"] == pced.AGG_MOE else (lw.exp() * p).sum(1)
        score, token = mixed.max(dim=1)
        expert = (lw + p).gather(2, token[:, None, None].expand(B, N, 1))[..., 0].max(dim=1)[1].int() + 1
    out = dict(hidden=h, lse=lse, score=score, seq_len=st["base"] + 1, step=torch.ones(1, dtype=torch.int32))
    if B == 1:
        out.update(token=token.int(), expert=expert)
    if c["first"]:
        out["beta"] = beta
    out["rows"] = [rows[:, :, s] for s in range(S)] if S <= 33 else rows
    return out
