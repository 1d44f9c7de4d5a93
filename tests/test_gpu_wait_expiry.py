"""Failure detection without a GPU fault: a bounded device-side wait that runs
out (a barrier nothing ever completes) must come back as an error status the
host can read, leave no hang behind, and leave the context usable."""
import time

import numpy as np
import pytest

from paper_2604_05650_b200 import workloads as W

pytestmark = pytest.mark.gpu


def test_expired_wait_is_reported_and_the_context_stays_usable(oracle_mod):
    import torch
    from paper_2604_05650_b200 import binding
    from gpu_util import run_attention, assert_attention_close
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    ctx = binding.Context(0)
    try:
        ctx.set_stream(torch.cuda.current_stream().cuda_stream)
        assert ctx.device_status_code() == (binding.OK, 0)
        t0 = time.perf_counter()
        ctx.selftest_wait_expiry(20)                      # gives up after 20 ms
        code, flags = ctx.device_status_code()            # synchronises the stream
        waited = time.perf_counter() - t0
        assert code == binding.ERR_TIMEOUT and flags & binding.DEV_WAIT_EXPIRED
        assert 0.015 <= waited < 1.5, waited
        assert ctx.device_status_code() == (binding.OK, 0)   # reported once, then cleared
        # the context and the device still work
        cfg = W.sweep_config(gamma=4, kv_len=2048, batch=1)
        case = W.attention_inputs(cfg)
        out, mass = run_attention(ctx, *case)
        ref_out, ref_mass = oracle_mod.verify_attention(*case)
        assert_attention_close(out, mass, ref_out, ref_mass)
        with pytest.raises(binding.LvspecError):
            ctx.selftest_wait_expiry(0)
    finally:
        ctx.close()


@pytest.mark.parametrize("polls", [None, 0])
def test_calls_after_an_expired_wait_are_right(polls, monkeypatch):
    """An expired wait may leave words in the buffer through which the splits' partials go.  The calls
    after it must not take them for their own, whether or not the status has been read."""
    import torch
    from paper_2604_05650_b200 import binding
    from gpu_util import dev_bf16
    if polls is not None:
        monkeypatch.setenv("LVSPEC_MERGE_POLLS", str(polls))
    ctx = binding.Context(0)
    ctx.set_stream(torch.cuda.current_stream().cuda_stream)
    calls = []
    # the widest merging launch first; (KV heads, G, gamma, D, length, splits)
    for hkv, G, gamma, D, L, ns in ((4, 7, 8, 128, 4113, 32), (2, 8, 9, 128, 900, 6), (2, 4, 4, 64, 1024, 8)):
        rng = np.random.default_rng(ns)
        bf = lambda *s: dev_bf16(W.f32_to_bf16_bits(rng.standard_normal(s).astype(np.float32)))
        calls.append((binding.attn_shape(1, gamma, hkv * G, hkv, D, L, ns),
                      bf(1, gamma, hkv * G, D), bf(1, hkv, L, D), bf(1, hkv, L, D), [L], [[9, L // 2]]))

    def results():
        res = []
        for shape, q, k, v, lens, span in calls:       # one after the other, no synchronisation between
            out, mass = torch.empty_like(q), torch.empty(q.shape[:3], device="cuda")
            ctx.verify_attention(shape, q, k, v, lens, span, out, mass)
            res += [out, mass]
        return res

    try:
        first = results()
        assert ctx.device_status_code() == (binding.OK, 0)
        assert all(torch.isfinite(x.float()).all() for x in first)
        ctx.selftest_wait_expiry(1)
        for _ in range(5):
            for a, b in zip(first, results()):
                assert torch.equal(a, b)
        assert ctx.device_status_code() == (binding.ERR_TIMEOUT, binding.DEV_WAIT_EXPIRED)
        before = ctx.launch_count()
        for _ in range(5):
            for a, b in zip(first, results()):
                assert torch.equal(a, b)
        assert ctx.launch_count() - before == 5 * len(calls)       # all of them merge inside the launch
        assert ctx.device_status_code() == (binding.OK, 0)
    finally:
        ctx.close()


def test_reading_the_status_leaves_nothing_on_the_stream():
    """A caller may go on on another stream once the status has been read: what the reading puts in
    order is in order by then."""
    import torch
    from paper_2604_05650_b200 import binding
    ctx = binding.Context(0)
    stream = torch.cuda.Stream()
    ctx.set_stream(stream)
    try:
        for _ in range(20):
            ctx.selftest_wait_expiry(1)
            assert ctx.device_status_code() == (binding.ERR_TIMEOUT, binding.DEV_WAIT_EXPIRED)
            assert stream.query()
    finally:
        ctx.close()
