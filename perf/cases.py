"""What is timed when this library's speed is measured: whole verify steps, as a decoding
loop runs them through ``paper_2604_05650_b200.binding``.

A ``step`` case is one pass of the verify step over all layers of a target model: one
attention call per layer on that layer's own KV cache, then the acceptance pass with the
emit step on the target logits, judged on the last layer's visual mass.  A ``score`` case
is the paper's own relevance score (Eq. 4) followed by the acceptance pass on it, with or
without the one-off norms of the visual hidden states that follow prefill.  Calls go out
one after the other, as a decoding loop makes them (lengths change from step to step, so
they are arguments of every call); nothing is synchronised inside a pass.

Shapes are those of ``workloads.CONFIGS`` and its head-shape sweep, of the tests, or
generic.  Values follow the input recipe of ``workloads``: N(0, 1) hidden values, visual
keys shifted by +0.5 on eight channels per KV head, logits N(0, 3) with one planted token
per row.  One thing is added: the draft positions differ in how visual they are, as the
paper's premise has it (their queries lean towards or away from the visual keys' shift by
position), so the ranking of their scores does not hang on the last bits of a sum.
"""
import math

import torch

from paper_2604_05650_b200 import binding

# (query heads, KV heads, head_dim): the Qwen2.5-VL-7B / -32B, LLaVA-OneVision-72B shaped
# configurations and the tiny one
HEADS = ((28, 4, 128), (40, 8, 128), (64, 8, 128), (8, 2, 64))
VOCAB = 152064
GIB = 1 << 30


def _step(name, heads, layers, batch, gamma, kv_len, visual_start, visual_len, *, cache="dense", branches=1,
          frames=1, page=0, ragged=False, vocab=VOCAB, window=None):
    """cache: "dense" [B, Hkv, L, D], "position" [B, L, Hkv, D], "paged", "fp8".  gamma counts
    the draft tokens of one branch.  frames > 1: the visual tokens come in that many spans
    with three text tokens between two, and the last layer's call takes all the spans."""
    hq, hkv, d = heads
    case = {"kind": "step", "hq": hq, "hkv": hkv, "d": d, "layers": layers, "batch": batch, "gamma": gamma,
            "branches": branches, "kv_len": kv_len, "visual_start": visual_start, "visual_len": visual_len,
            "frames": frames, "cache": cache, "page": page, "ragged": ragged, "vocab": vocab,
            "window": gamma if window is None else window, "lam": 0.7}
    return dict(case, name=name) if name else case


def _score(name, batch, gamma, n_visual, dim, top_n, prefill, vocab=VOCAB):
    case = {"kind": "score", "batch": batch, "gamma": gamma, "n_visual": n_visual, "dim": dim, "top_n": top_n,
            "prefill": prefill, "vocab": vocab, "window": gamma, "lam": 0.7}
    return dict(case, name=name) if name else case


def listed():
    return [
        # the smallest call there is: one short head_dim 64 layer and a small vocabulary, all latency
        _step("tiny", HEADS[3], 1, 1, 4, 1024, 64, 768, vocab=4096, window=1),
        # a few frames and a short prompt, on the position-major cache of most model code
        _step("short-clip", HEADS[1], 16, 1, 4, 4096, 256, 3072, cache="position"),
        # 7B target, 64 sampled frames with a time stamp between two (the mass is taken over all of them)
        _step("7b-frames", HEADS[0], 28, 1, 8, 16384, 256, 64 * 196, frames=64),
        # 32B target, 128 frames, a chain of 8: the shape the library is quoted on
        _step("32b-chain", HEADS[1], 64, 1, 8, 32768, 512, 128 * 196),
        # 72B target: 80 query rows per KV head
        _step("72b-chain", HEADS[2], 80, 1, 10, 32768, 512, 32 * 729),
        # 32B target on an 8-bit cache
        _step("32b-fp8", HEADS[1], 64, 1, 8, 32768, 512, 128 * 196, cache="fp8"),
        # 32B target, the draft tree of the paper's appendix: two branches of 10 tokens
        _step("32b-tree", HEADS[1], 32, 1, 10, 32768, 512, 128 * 196, branches=2),
        # a serving engine: four requests of different lengths on a paged cache
        _step("serve-paged", HEADS[1], 16, 4, 8, 20480, 320, 15000, cache="paged", page=512, ragged=True),
        # sixteen requests of different odd lengths in one batch
        _step("serve-batch", HEADS[1], 4, 16, 8, 15999, 256, 12001, ragged=True),
        # hours of video: four sequences of 128 K positions, long drafts
        _step("long-video", HEADS[1], 2, 4, 16, 131072, 256, 98304),
        # the paper's own score in every step: 25088 visual tokens against 8 draft tokens, N = 10
        _score("score-step", 1, 8, 128 * 196, 5120, 10, False),
        # the first step after prefill: the visual rows' norms too; 72B shape, N = 100 of the sensitivity table
        _score("score-prefill", 1, 10, 32 * 729, 8192, 100, True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    if rng.random() < 0.15:
        batch = rng.choice((1, 1, 2, 4))
        dim = 64 * _log_int(rng, 8, 128)
        n_visual = min(_log_int(rng, 500, 40000), GIB // (2 * dim * batch))
        return _score(None, batch, rng.randint(2, 16), n_visual, dim, rng.choice((1, 5, 10, 10, 32, 100)),
                      rng.random() < 0.3, rng.choice((VOCAB, 32000)))
    cache = rng.choice(("dense", "dense", "dense", "position", "paged", "fp8", "tree", "frames"))
    heads = rng.choice(HEADS[:3] if cache in ("paged", "fp8") or rng.random() < 0.9 else HEADS[3:])
    hq, hkv, d = heads
    branches = 2 if cache == "tree" else 1
    most = (80 if cache == "fp8" else 128) // (hq // hkv) // branches
    gamma = rng.randint(2, min(16, most))
    batch = rng.choice((1, 1, 1, 2, 3, 4, 8, 16))
    kv_len = _log_int(rng, 1000, 131072)
    page = 0
    if cache == "paged":
        page = rng.choice((128, 256, 512, 1024))
    esz = 1 if cache == "fp8" else 2
    per_layer = 2 * batch * hkv * kv_len * d * esz
    while per_layer > 4 * GIB:
        kv_len //= 2
        per_layer //= 2
    # as many layers as a model has, within 4 GiB of cache
    layers = max(1, min(_log_int(rng, 8, 80), 4 * GIB // per_layer))
    visual_start = rng.randint(0, kv_len // 20)
    visual_len = int((kv_len - visual_start - gamma * branches) * rng.uniform(0.5, 0.9))
    frames = 1
    if cache == "frames":
        frames = rng.randint(2, max(2, min(128, visual_len // 64)))
        visual_len -= 3 * frames
    return _step(None, heads, layers, batch, gamma, kv_len, visual_start, visual_len,
                 cache="dense" if cache in ("tree", "frames") else cache, branches=branches, frames=frames, page=page,
                 ragged=batch > 1 and rng.random() < 0.7, vocab=rng.choice((VOCAB, VOCAB, 32000, 50257)))


# ---------------------------------------------------------------- lengths and spans
def _lengths(case):
    """kv_len of every sequence: a ragged batch runs down to about half the longest."""
    n, longest = case["batch"], case["kv_len"]
    if not case["ragged"]:
        return [longest] * n
    return [longest - b * longest // (2 * n) - (b * 37) % 61 for b in range(n)]


def _spans(case):
    """Per sequence the visual spans [start, end), `frames` of them."""
    out = []
    for length in _lengths(case):
        start = case["visual_start"] * length // case["kv_len"]
        total = case["visual_len"] * length // case["kv_len"]
        n = case["frames"]
        each, spans, pos = total // n, [], start
        for i in range(n):
            size = each + (1 if i < total - each * n else 0)
            spans.append([pos, pos + size])
            pos += size + 3
        out.append(spans)
    return out


def _capacity(case):
    """Cache slots per sequence: whole pages on a paged cache, else the longest sequence."""
    page = case["page"]
    return -(-case["kv_len"] // page) * page if page else case["kv_len"]


# ---------------------------------------------------------------- inputs
def _normal(shape, gen, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(generator=gen)


def _accept_inputs(case, rows, gamma, gen):
    """Target logits [rows, gamma, V] and draft tokens: 40 % the row's target token, 25 % a
    neighbour's, the rest random."""
    vocab = case["vocab"]
    logits = _normal((rows, gamma, vocab), gen, torch.float32).mul_(3.0)
    planted = torch.randint(0, vocab, (rows, gamma, 1), generator=gen, device="cuda")
    logits.scatter_add_(2, planted, torch.full((rows, gamma, 1), 8.0, device="cuda"))
    top = logits.argmax(-1)
    kind = torch.rand((rows, gamma), generator=gen, device="cuda")
    draft = torch.where(kind < 0.4, top, torch.where(kind < 0.65, top.roll(1, 1),
                                                     torch.randint(0, vocab, (rows, gamma), generator=gen, device="cuda")))
    return logits, draft.to(torch.int32).contiguous()


def _new(shape, dtype):
    return torch.zeros(shape, dtype=dtype, device="cuda")


def _emit_buffers(rows, gamma):
    return {"accept_len": _new((rows,), torch.int32), "emitted": _new((rows, gamma), torch.int32),
            "n_emitted": _new((rows,), torch.int32), "new_kv_len": _new((rows,), torch.int32)}


def _context():
    ctx = binding.Context(torch.cuda.current_device())
    ctx.set_stream(torch.cuda.current_stream())
    return ctx


def _prepare_score(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    batch, gamma, lv, dim = case["batch"], case["gamma"], case["n_visual"], case["dim"]
    hv = _normal((batch, lv, dim), gen)
    hd = _normal((batch, gamma, dim), gen)
    # every draft token is drawn to a few salient visual tokens, each more than the one before
    for b in range(batch):
        for k in range(gamma):
            rows = torch.randint(0, lv, (8,), generator=gen, device="cuda")
            hd[b, k] += (0.1 + 0.8 * k / gamma) * hv[b, rows].float().sum(0).to(torch.bfloat16)
    order = torch.randperm(gamma, generator=gen, device="cuda")
    hd = hd[:, order].contiguous()
    logits, draft = _accept_inputs(case, batch, gamma, gen)
    ctx = _context()
    inv = _new((batch, lv), torch.float32)
    ctx.row_inv_norms(batch * lv, dim, hv, inv)
    ctx.reserve(max(ctx.relevance_workspace_bytes(batch, gamma, lv, dim),
                    ctx.accept_workspace_bytes(batch, gamma, case["vocab"])))
    return {"case": case, "ctx": ctx, "hv": hv, "hd": hd, "inv": inv, "logits": logits, "draft": draft,
            "relevance": _new((batch, gamma), torch.float32),
            "kv_len": torch.full((batch,), lv + 512, dtype=torch.int32, device="cuda"), **_emit_buffers(batch, gamma)}


def _prepare_step(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    hq, hkv, d, layers, batch = case["hq"], case["hkv"], case["d"], case["layers"], case["batch"]
    queries = case["gamma"] * case["branches"]
    lengths, spans, cap, page, cache = _lengths(case), _spans(case), _capacity(case), case["page"], case["cache"]
    # the eight channels of every KV head on which visual keys are shifted
    dims = torch.stack([torch.randperm(d, generator=gen, device="cuda")[:8] for _ in range(hkv)])
    shift = torch.zeros((hkv, d), device="cuda").scatter_(1, dims, 0.5)
    # how far a draft position's queries lean towards it, in shuffled order
    lean = torch.linspace(-2.0, 2.0, queries, device="cuda")[torch.randperm(queries, generator=gen, device="cuda")]
    q_shift = (2.0 * lean[:, None, None] * shift.repeat_interleave(hq // hkv, 0)).to(torch.bfloat16)
    shift = shift.to(torch.bfloat16)
    q = [_normal((batch, queries, hq, d), gen).add_(q_shift) for _ in range(layers)]
    hull = [[s[0][0], s[-1][1]] for s in spans]
    state = {"case": case, "q": q, "kv_len": lengths, "span": hull, "spans": spans}
    k, v, k_scale, v_scale = [], [], [], []
    if cache == "paged":
        per_seq = cap // page
        pages = batch * per_seq
        table = torch.randperm(pages, generator=gen, device="cuda").to(torch.int32).view(batch, per_seq)
        state["table"], state["n_pages"] = table, pages
    for _ in range(layers):
        if cache == "paged":
            kk, vv = _normal((pages, hkv, page, d), gen), _normal((pages, hkv, page, d), gen)
            for b in range(batch):
                visual = torch.zeros(cap, dtype=torch.bfloat16, device="cuda")
                visual[hull[b][0]:hull[b][1]] = 1
                kk[table[b].long()] += visual.view(per_seq, 1, page, 1) * shift[:, None, :]
        elif cache == "position":
            kk, vv = _normal((batch, cap, hkv, d), gen), _normal((batch, cap, hkv, d), gen)
            for b in range(batch):
                kk[b, hull[b][0]:hull[b][1]] += shift
        else:
            kk, vv = _normal((batch, hkv, cap, d), gen), _normal((batch, hkv, cap, d), gen)
            for b in range(batch):
                kk[b, :, hull[b][0]:hull[b][1]] += shift[:, None, :]
        if cache == "fp8":
            for x, codes, scales in ((kk, k, k_scale), (vv, v, v_scale)):
                scale = x.abs().amax((2, 3)).float().clamp_(min=1e-6) / 448.0
                codes.append((x / scale[:, :, None, None]).to(torch.float8_e4m3fn).view(torch.uint8))
                scales.append(scale)
        else:
            k.append(kk)
            v.append(vv)
    state.update(k=k, v=v, k_scale=k_scale, v_scale=v_scale)
    rows = batch * case["branches"]
    logits, draft = _accept_inputs(case, rows, case["gamma"], gen)
    ctx = _context()
    shape = binding.attn_shape(batch, queries, hq, hkv, d, cap)
    ctx.reserve(max(ctx.attention_workspace_bytes(shape, max(lengths)),
                    ctx.accept_workspace_bytes(rows, case["gamma"], case["vocab"])))
    state.update(ctx=ctx, shape=shape, logits=logits, draft=draft, out=_new((layers, batch, queries, hq, d), torch.bfloat16),
                 mass=_new((layers, batch, queries, hq), torch.float32),
                 kv_len_dev=torch.tensor(lengths, dtype=torch.int32, device="cuda").repeat_interleave(case["branches"]),
                 **_emit_buffers(rows, case["gamma"]))
    # a program holds each layer's buffers by themselves
    state["out_l"], state["mass_l"] = list(state["out"]), list(state["mass"])
    state["strides"] = (cap * hkv * d, d, hkv * d)
    if case["branches"] > 1:
        state.update(best_branch=_new((batch,), torch.int32), best_len=_new((batch,), torch.int32))
    return state


def prepare(case, seed):
    return (_prepare_score if case["kind"] == "score" else _prepare_step)(case, seed)


# ---------------------------------------------------------------- one pass
def _run_score(s):
    c, ctx = s["case"], s["ctx"]
    batch, gamma = c["batch"], c["gamma"]
    if c["prefill"]:
        ctx.row_inv_norms(batch * c["n_visual"], c["dim"], s["hv"], s["inv"])
    ctx.visual_relevance(batch, gamma, c["n_visual"], c["dim"], s["hd"], s["hv"], s["inv"], c["top_n"], s["relevance"])
    ctx.loose_accept_emit(batch, gamma, c["vocab"], 1, s["logits"], s["draft"], s["relevance"], s["accept_len"],
                          s["emitted"], s["n_emitted"], c["window"], lam=c["lam"], kv_len=s["kv_len"],
                          new_kv_len=s["new_kv_len"])
    return [s["inv"], s["relevance"], s["accept_len"], s["emitted"], s["n_emitted"], s["new_kv_len"]]


def _run_step(s):
    c, ctx, shape, cache = s["case"], s["ctx"], s["shape"], s["case"]["cache"]
    q, k, v, out, mass, kv_len, span = s["q"], s["k"], s["v"], s["out_l"], s["mass_l"], s["kv_len"], s["span"]
    last = c["layers"] - 1
    for i in range(c["layers"]):
        if i == last and c["frames"] > 1:
            ctx.verify_attention_spans(shape, q[i], k[i], v[i], kv_len, s["spans"], out[i], mass[i])
        elif c["branches"] > 1:
            ctx.verify_attention_tree(shape, c["branches"], q[i], k[i], v[i], kv_len, span, out[i], mass[i])
        elif cache == "fp8":
            ctx.verify_attention_fp8(shape, q[i], k[i], v[i], s["k_scale"][i], s["v_scale"][i], kv_len, span,
                                     out[i], mass[i])
        elif cache == "paged":
            ctx.verify_attention_paged(shape, c["page"], s["n_pages"], q[i], k[i], v[i], s["table"], kv_len, span,
                                       out[i], mass[i])
        elif cache == "position":
            ctx.verify_attention_strided(shape, s["strides"], s["strides"], q[i], k[i], v[i], kv_len, span,
                                         out[i], mass[i])
        else:
            ctx.verify_attention(shape, q[i], k[i], v[i], kv_len, span, out[i], mass[i])
    rows = c["batch"] * c["branches"]
    ctx.loose_accept_emit(rows, c["gamma"], c["vocab"], c["hq"], s["logits"], s["draft"], mass[last], s["accept_len"],
                          s["emitted"], s["n_emitted"], c["window"], lam=c["lam"], kv_len=s["kv_len_dev"],
                          new_kv_len=s["new_kv_len"])
    got = [s["out"], s["mass"], s["accept_len"], s["emitted"], s["n_emitted"], s["new_kv_len"]]
    if c["branches"] > 1:
        ctx.select_branch(c["batch"], c["branches"], s["accept_len"], s["best_branch"], s["best_len"])
        got += [s["best_branch"], s["best_len"]]
    return got


def run(state):
    return (_run_score if state["case"]["kind"] == "score" else _run_step)(state)


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    rows = case["batch"] * case.get("branches", 1) * case["gamma"]
    bytes_ = rows * case["vocab"] * 4 + rows * 8          # logits, draft tokens and emitted tokens
    if case["kind"] == "score":
        visual = case["batch"] * case["n_visual"]
        bytes_ += visual * (case["dim"] * 2 + 4) + rows * (case["dim"] * 2 + 4)
        flops = 2 * rows * case["n_visual"] * case["dim"] + (2 * visual * case["dim"] if case["prefill"] else 0)
        return {"bytes": bytes_, "flops": flops}
    hq, hkv, d, positions = case["hq"], case["hkv"], case["d"], sum(_lengths(case))
    esz = 1 if case["cache"] == "fp8" else 2
    queries = case["gamma"] * case["branches"]
    per_layer = 2 * hkv * positions * d * esz + rows * hq * (2 * d * 2 + 4)
    return {"bytes": bytes_ + case["layers"] * per_layer, "flops": case["layers"] * 4 * queries * hq * d * positions}


def tolerance(case):
    # About four times what the calls differ by from the operation in 64 bits on the same
    # inputs: norms and scores 8e-6 (fp32 sums of up to 8192 products), largest 9e-6; attention
    # 2.4e-3 (bf16 probabilities and results), largest 1.3e-2.  Masses are closer than that
    # (5e-5, largest 2e-4); tokens and lengths are the same.
    if case["kind"] == "score":
        return {"rel": 3e-5, "max": 1e-4}
    return {"rel": 1e-2, "max": 5e-2}
