"""Merge of the splits inside the attention kernel: a head of 2 to 32 splits whose CTAs all run at
once, at most twelve rows a split.  On both sides of each limit against the oracle; and with
LVSPEC_MERGE_POLLS=0, where every CTA that would have to wait gives its share to the last one to
arrive, the same bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# name: (B, Hkv, G, gamma, D, lengths, n_split); a launch merges its splits itself where it holds
# B * Hkv * n_split <= SMs, n_split <= 32 and rows <= 12 * splits that have a tile
CASES = {
    "two-splits": ((1, 2, 2, 3, 128, [700], 2), True),
    "rows-12-a-split": ((1, 2, 8, 9, 128, [900], 6), True),
    "rows-13-a-split": ((1, 2, 6, 13, 128, [900], 6), False),
    "128-rows": ((1, 1, 8, 16, 128, [3000], 11), True),
    "three-warps-idle": ((1, 1, 5, 1, 128, [2500], 4), True),
    "more-splits-than-rows": ((1, 2, 1, 3, 64, [4000], 31), True),
    "32-splits": ((1, 4, 7, 8, 128, [4096 + 17], 32), True),
    "33-splits": ((1, 2, 5, 4, 128, [4400], 33), False),
    "splits-without-tiles": ((2, 2, 4, 5, 128, [2500, 300], 18), True),
    "rows-of-the-shortest": ((2, 2, 5, 8, 128, [2500, 300], 18), False),
    "head-dim-64": ((1, 2, 4, 4, 64, [1024], 8), True),
}


def _inputs(case, seed):
    from paper_2604_05650_b200 import workloads as W
    B, hkv, G, gamma, D, lens, ns = case
    rng = np.random.default_rng(seed)
    bf = lambda *s: W.f32_to_bf16_bits(rng.standard_normal(s).astype(np.float32))
    cap = max(lens) + 5
    q, k, v = bf(B, gamma, hkv * G, D), bf(B, hkv, cap, D), bf(B, hkv, cap, D)
    return q, k, v, np.array(lens, np.int32), np.array([[n // 7, n // 2] for n in lens], np.int32), ns


def _contexts(monkeypatch, polls=None):
    from paper_2604_05650_b200 import binding
    if polls is not None:
        monkeypatch.setenv("LVSPEC_MERGE_POLLS", str(polls))
    ctx = binding.Context(0)
    monkeypatch.delenv("LVSPEC_MERGE_POLLS", raising=False)
    return ctx


@pytest.mark.parametrize("name", CASES)
def test_both_sides_of_each_limit(name, oracle_mod, monkeypatch):
    from gpu_util import assert_attention_close, run_attention
    case, merged = CASES[name]
    q, k, v, lens, span, ns = _inputs(case, 17)
    ref = oracle_mod.verify_attention(q, k, v, lens, span)
    waiting, giving_up = _contexts(monkeypatch), _contexts(monkeypatch, 0)
    before = waiting.launch_count()
    first = run_attention(waiting, q, k, v, lens, span, ns)
    assert waiting.launch_count() - before == (1 if merged else 2)
    assert_attention_close(*first, *ref)
    # the exchange buffer is as it was: other shapes and the same one again, on both contexts
    others = [_inputs(c, 3) for c, m in CASES.values() if m]
    for ctx in (waiting, giving_up):
        for _ in range(20):
            out, mass = run_attention(ctx, q, k, v, lens, span, ns)
            assert (out == first[0]).all() and (mass == first[1]).all()
            for o in others[:4]:
                run_attention(ctx, *o)
        ctx.close()


def test_two_contexts_share_the_gpu(monkeypatch):
    """Attention calls of two contexts on two streams: grids whose CTAs may get SMs in any order.  (No
    grid waits for another: a CTA that waits in vain leaves after some 40 us.)"""
    import torch
    from gpu_util import dev_bf16
    from paper_2604_05650_b200 import binding
    case = (1, 8, 5, 8, 128, [16384], 16)
    q, k, v, lens, span, ns = _inputs(case, 5)
    B, hkv, G, gamma, D = case[:5]
    dq, dk, dv = dev_bf16(q), dev_bf16(k), dev_bf16(v)
    shape = binding.attn_shape(B, gamma, hkv * G, hkv, D, k.shape[2], ns)
    streams, ctxs, outs = [torch.cuda.Stream() for _ in range(2)], [], []
    for s in streams:
        ctxs.append(_contexts(monkeypatch))
        ctxs[-1].set_stream(s)
        outs.append([(torch.empty_like(dq), torch.empty((B, gamma, hkv * G), device="cuda")) for _ in range(40)])
    torch.cuda.synchronize()
    for i in range(40):
        for ctx, o in zip(ctxs, outs):
            ctx.verify_attention(shape, dq, dk, dv, lens, span, *o[i])
    torch.cuda.synchronize()
    for ctx, o in zip(ctxs, outs):
        assert ctx.device_status() == 0
        for out, mass in o:
            assert torch.equal(out, outs[0][0][0]) and torch.equal(mass, outs[0][0][1])
        ctx.close()


@pytest.mark.parametrize("name", [n for n, (c, merged) in CASES.items() if merged])
def test_on_a_shared_gpu_a_kernel_merges(name, oracle_mod, monkeypatch):
    from gpu_util import assert_attention_close, run_attention
    q, k, v, lens, span, ns = _inputs(CASES[name][0], 29)
    ref = oracle_mod.verify_attention(q, k, v, lens, span)
    ctx = _contexts(monkeypatch)
    for shared, launches in ((True, 2), (False, 1), (True, 2)):
        ctx.set_gpu_shared(shared)
        before = ctx.launch_count()
        got = run_attention(ctx, q, k, v, lens, span, ns)
        assert ctx.launch_count() - before == launches
        assert_attention_close(*got, *ref)
    ctx.close()


def _forms():
    """Every form of the call that can merge inside its launch, on 16 splits of 17 tiles (so that most CTAs
    of a head have to wait for one): name -> call(ctx) giving (out, mass)."""
    import torch
    from gpu_util import dev_bf16
    from paper_2604_05650_b200 import binding
    from paper_2604_05650_b200 import workloads as W
    L, hkv, G, gamma, ns = 17 * 128, 8, 5, 8, 16
    q, k, v, lens, span, _ = _inputs((1, hkv, G, gamma, 128, [L], ns), 41)
    k, v = k[:, :, :L], v[:, :, :L]
    dq, dk, dv = dev_bf16(q), dev_bf16(k), dev_bf16(v)
    (k8, ks), (v8, vs) = W.quantize_cache_e4m3(k), W.quantize_cache_e4m3(v)
    d8 = [torch.from_numpy(x).cuda() for x in (k8, v8, ks, vs)]
    spans = np.array([[[5, 100], [130, 131], [300, 1900]]], np.int32)
    table = torch.arange(17, dtype=torch.int32, device="cuda").flip(0).contiguous()[None]
    pool = lambda x: x[0].reshape(hkv, 17, 128, 128).permute(1, 0, 2, 3).flip(0).contiguous()
    pk, pv = pool(dk), pool(dv)
    by_pos = [x.permute(0, 2, 1, 3).contiguous() for x in (dk, dv)]
    st = (L * hkv * 128, 128, hkv * 128)
    shape = binding.attn_shape(1, gamma, hkv * G, hkv, 128, L, ns)
    short = lens.tolist(), span.tolist()

    def call(name):
        def go(ctx):
            out, mass = torch.full_like(dq, float("nan")), torch.full((1, gamma, hkv * G), float("nan"), device="cuda")
            ctx.set_stream(torch.cuda.current_stream())
            if name == "fp8":
                ctx.verify_attention_fp8(shape, dq, *d8, *short, out, mass)
            elif name == "spans":
                ctx.verify_attention_spans(shape, dq, dk, dv, lens, spans, out, mass)
            elif name == "paged":
                ctx.verify_attention_paged(shape, 128, 17, dq, pk, pv, table, *short, out, mass)
            elif name == "strided":
                ctx.verify_attention_strided(shape, st, st, dq, *by_pos, *short, out, mass)
            elif name == "tree":
                ctx.verify_attention_tree(shape, 2, dq, dk, dv, *short, out, mass)
            else:
                ctx.verify_attention(shape, dq, dk, dv, *short, out, mass)
            return out, mass
        return go
    return {name: call(name) for name in ("dense", "fp8", "spans", "paged", "strided", "tree")}


@pytest.mark.parametrize("name", ["dense", "fp8", "spans", "paged", "strided", "tree"])
def test_shares_given_up_are_merged_alike(name, monkeypatch):
    """The path of a CTA that waits in vain is really taken (another stream's matrix products let the CTAs of a
    launch start at different times), and its results are the same bits."""
    import torch
    call = _forms()[name]
    waiting, giving_up = _contexts(monkeypatch), _contexts(monkeypatch, 0)
    try:
        first = call(waiting)
        assert all(torch.isfinite(x.float()).all() for x in first)
        side, x = torch.cuda.Stream(), torch.randn(4096, 4096, device="cuda").bfloat16()
        x @ x
        torch.cuda.synchronize()
        for _ in range(20):
            with torch.cuda.stream(side):
                x @ x, x @ x
            got = [call(giving_up) for _ in range(5)]
            for out, mass in got:
                assert torch.equal(out, first[0]) and torch.equal(mass, first[1])
        assert giving_up.merge_handed_over() > 0
        assert waiting.device_status() == 0 and giving_up.device_status() == 0
    finally:
        waiting.close()
        giving_up.close()


BAD = {"nan": 0x7FC0, "nan-all-ones": 0xFFFF, "inf": 0x7F80, "minus-inf": 0xFF80}


@pytest.mark.parametrize("polls", [None, 0])
@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("where", ["q", "k", "v"])
def test_not_a_number_goes_through(where, bad, polls, monkeypatch):
    """NaN and infinities among the inputs: no reader waits for a word in vain, and the results are those of the
    merge kernel.  A finite result is a sum of the same partials in another order: fp32 roundings, and at
    most one bf16 step (2^-7 of the value) where they straddle a rounding boundary."""
    import torch
    from gpu_util import dev_bf16
    from paper_2604_05650_b200 import binding
    (B, hkv, G, gamma, D), L, ns = (1, 2, 5, 8, 128), 2000, 8
    q, k, v, lens, span, _ = _inputs((B, hkv, G, gamma, D, [L], ns), 43)
    x = {"q": q[:, 3, 2], "k": k[:, 1, 700], "v": v[:, 1, [0, 900, L - 1]]}[where]
    x[..., 5] = BAD[bad]
    if where == "v":
        v[:, 1, [0, 900, L - 1]] = x
    dq, dk, dv = dev_bf16(q), dev_bf16(k), dev_bf16(v)
    shape = binding.attn_shape(B, gamma, hkv * G, hkv, D, k.shape[2], ns)
    ctx = _contexts(monkeypatch, polls)
    ctx.set_stream(torch.cuda.current_stream())
    res = []
    for shared in (True, False, False):
        ctx.set_gpu_shared(shared)
        out, mass = torch.empty_like(dq), torch.empty((B, gamma, hkv * G), device="cuda")
        ctx.verify_attention(shape, dq, dk, dv, lens, span, out, mass)
        res.append((out.float(), mass))
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    ctx.close()
    (ref_o, ref_m), (o, m), again = res
    assert torch.equal(o.view(torch.int32), again[0].view(torch.int32)) and torch.equal(m.view(torch.int32), again[1].view(torch.int32))
    assert torch.isfinite(ref_o).any()
    for a, b, step in ((ref_o, o, 2.0 ** -7), (ref_m, m, 1e-5)):
        assert torch.equal(torch.isnan(a), torch.isnan(b)) and torch.equal(torch.isinf(a), torch.isinf(b))
        assert torch.equal(a[torch.isinf(a)], b[torch.isinf(b)])
        fin = torch.isfinite(a)
        assert ((a - b).abs()[fin] <= step * a.abs()[fin] + 1e-6).all()
