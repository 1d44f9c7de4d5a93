"""A batch whose sequences differ in length may be cut for two waves of CTAs (n_split 0).  Every
entry point, in two waves: the library's own choice gives bit for bit what that split count
gives when asked for, and not what the count of one wave gives; parity with the oracle; and
the figure of the workspace query covers it."""
import numpy as np
import pytest

import test_gpu_attention as A
import test_gpu_fp8 as F8
import test_gpu_paged as PG
import test_gpu_spans as SP
import test_gpu_strided as ST
import test_gpu_tree as TR

pytestmark = pytest.mark.gpu

B, HKV, LMAX = 8, 8, 3072
KV_LEN = [3000] + [200 + 7 * b for b in range(B - 1)]
SPAN = [[10, n - 30] for n in KV_LEN]


@pytest.fixture(scope="module")
def ctx():
    from paper_2604_05650_b200 import binding
    c = binding.Context(0)
    yield c
    c.close()


def _two_waves():
    import torch
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    return min(2 * n_sm // (B * HKV), (max(KV_LEN) + 127) // 128)


def _check(run, ref, splits_of_one_wave):
    from gpu_util import assert_attention_close
    two = _two_waves()
    assert two > splits_of_one_wave > 0
    out, mass = run(0)
    assert_attention_close(out, mass, *ref)
    out_2, mass_2 = run(two)
    assert (out == out_2).all() and (mass == mass_2).all()
    out_1, _ = run(max(2, splits_of_one_wave))
    assert (out != out_1).any()


def _np(pair):
    from gpu_util import bf16_to_f64
    return bf16_to_f64(pair[0]), pair[1].cpu().numpy().astype(np.float64)


FORMS = ["dense", "head_dim_64", "strided", "paged", "spans", "tree", "fp8"]
# 40, 80 and 104 rows per KV head (the fp8 cache takes up to 80)
CASES = [(form, gamma, hq) for form in FORMS for gamma, hq in ((8, 40), (8, 80), (13, 64))
         if form != "fp8" or gamma * hq <= 80 * HKV]


@pytest.mark.parametrize("form,gamma,hq", CASES, ids=[f"{f}-{g * h // HKV}" for f, g, h in CASES])
def test_every_entry_point(ctx, oracle_mod, form, gamma, hq):
    from gpu_util import dev_bf16, run_attention
    from paper_2604_05650_b200 import binding
    D = 64 if form == "head_dim_64" else 128
    one = ctx.attention_splits(binding.attn_shape(B, gamma, hq, HKV, D, LMAX), max(KV_LEN), fp8=form == "fp8")
    if form == "fp8":
        case = F8._case(71, B, gamma, hq, HKV, LMAX, KV_LEN, SPAN)
        _check(lambda n: F8.run_fp8(ctx, *case, n_split=n), oracle_mod.verify_attention_fp8(*case), one)
        return
    case = A._case(72, B, gamma, hq, HKV, D, LMAX, KV_LEN, SPAN)
    q, k, v, kv_len, span = case
    if form == "tree":
        # branches of half the drafts (an odd count: of one)
        branches = 2 if gamma % 2 == 0 else gamma
        ref = oracle_mod.verify_attention(*case, branch_len=gamma // branches)
        _check(lambda n: TR._run_tree(ctx, case, branches, 2, n)[:2], ref, one)
        return
    if form == "spans":
        spans = [[[10, 60], [70, n - 30]] for n in KV_LEN]
        ref = SP.oracle_union_mass(oracle_mod, q, k, v, kv_len, spans)
        _check(lambda n: SP.run_spans(ctx, q, k, v, kv_len, spans, n), ref, one)
        return
    ref = oracle_mod.verify_attention(*case)
    if form == "paged":
        k_pool, v_pool, table, n_pages = PG.scatter_pages(73, k, v, 256)
        run = lambda n: _np(PG.run_paged(ctx, q, k_pool, v_pool, table, n_pages, 256, LMAX, kv_len, span, n))
    elif form == "strided":
        kbuf, vbuf = (dev_bf16(x).permute(0, 2, 1, 3).contiguous() for x in (k, v))
        strides = (LMAX * HKV * D, D, HKV * D)
        run = lambda n: ST._run(ctx, q, kbuf, vbuf, strides, strides, (B, gamma, hq, HKV, D, LMAX), kv_len, span, 2, n)
    else:
        run = lambda n: run_attention(ctx, *case, n_split=n)
    _check(run, ref, one)


def test_one_split_per_head_becomes_two(oracle_mod):
    """96 units: one split each in one wave (the kernel normalises and writes itself), two waves
    make it three (two kernels); reserving the figure of the workspace query is enough."""
    from gpu_util import run_attention, assert_attention_close
    from paper_2604_05650_b200 import binding
    c = binding.Context(0)
    try:
        batch, kv_len = 12, [3000 - 230 * b for b in range(12)]
        case = A._case(61, batch, 2, 8, 8, 128, 3000, kv_len, [[10, n - 50] for n in kv_len])
        shape = binding.attn_shape(batch, 2, 8, 8, 128, 3000)
        assert c.attention_splits(shape, 3000) == 1
        c.reserve(c.attention_workspace_bytes(shape, 3000))
        cap = c.workspace_capacity()
        ref_out, ref_mass = oracle_mod.verify_attention(*case)
        out, mass = run_attention(c, *case)
        assert_attention_close(out, mass, ref_out, ref_mass)
        again, _ = run_attention(c, *case)
        assert (again == out).all() and c.workspace_capacity() == cap
        assert (run_attention(c, *case, n_split=3)[0] == out).all()
        assert (run_attention(c, *case, n_split=1)[0] != out).any()
    finally:
        c.close()
