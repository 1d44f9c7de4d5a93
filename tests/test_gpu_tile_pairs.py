"""bf16 cache: tiles go through the softmax stage in pairs where the buffers allow and a CTA
has many (from 17 tiles on up to 64 padded rows, from 5 on above, from 3 on at head_dim 64),
one by one elsewhere.  The sizes at which that can go wrong: odd and even tile counts per CTA
on both sides, a last tile that holds one position, draft slots across a tile boundary, every
number of column chunks per softmax group, streams long enough for the softmax stage to run
ahead of the P.V products by all its buffers, junk beyond kv_len."""
import numpy as np
import pytest

import test_gpu_attention as A

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2604_05650_b200 import binding
    c = binding.Context(0)
    yield c
    c.close()


def _junk_beyond(case, kv_len):
    """NaN and huge values in the slots at or beyond kv_len."""
    q, k, v, lens, span = case
    k, v = k.copy(), v.copy()
    for b, n in enumerate(kv_len):
        k[b, :, n:] = 0x7F7F
        v[b, :, n:] = 0x7FC0
    return q, k, v, lens, span


@pytest.mark.parametrize("rows", [(2, 8, 1), (8, 40, 8), (8, 28, 4), (10, 64, 8), (12, 64, 8), (13, 64, 8), (15, 64, 8), (16, 64, 8)],
                         ids=["16", "40", "56", "80", "96", "104", "120", "128"])
@pytest.mark.parametrize("tiles", [1, 2, 3, 4, 5, 8, 9, 16, 17])
def test_tiles_per_cta(ctx, oracle_mod, rows, tiles, head_dim=128):
    gamma, hq, hkv = rows
    hq, hkv = hq // hkv, 1                               # one KV head: the same rows
    lmax = 128 * tiles * 2
    # one split of all tiles less one position's worth; the draft slots straddle a boundary
    kv_len = [128 * (tiles - 1) + 1 + gamma // 2 if tiles > 1 else 128, lmax - 127]
    kv_len = [max(n, gamma) for n in kv_len]
    span = [[0, n - gamma] for n in kv_len]
    case = _junk_beyond(A._case(900 + tiles, 2, gamma, hq, hkv, head_dim, lmax, kv_len, span), kv_len)
    A._check(ctx, oracle_mod, case, n_split=1, kernel=2)
    A._check(ctx, oracle_mod, case, n_split=2, kernel=2)


@pytest.mark.parametrize("rows", [(8, 8, 2), (9, 64, 8), (15, 64, 8), (16, 64, 8)], ids=["32", "72", "120", "128"])
@pytest.mark.parametrize("tiles", [1, 2, 3, 5])
def test_tiles_per_cta_at_head_dim_64(ctx, oracle_mod, rows, tiles):
    test_tiles_per_cta(ctx, oracle_mod, rows, tiles, head_dim=64)


@pytest.mark.parametrize("ring", ["2,2,4,4", "2,2,2,4", "2,2,3,3", "2,2,2,2", "2,3,1,2", "1,1,1,2"])
def test_buffer_counts(ctx, oracle_mod, monkeypatch, ring):
    """A long single split (odd length) under other buffer counts: pairs and one by one."""
    monkeypatch.setenv("LVSPEC_TC_RING", ring)
    kv_len = [128 * 37 + 63]
    case = _junk_beyond(A._case(77, 1, 8, 10, 2, 128, 128 * 38, kv_len, [[130, 4000]]), kv_len)
    for _ in range(3):
        A._check(ctx, oracle_mod, case, n_split=1, kernel=2)


@pytest.mark.parametrize("ring", ["2,5,1,2", "2,8,1,2", "2,8,2,4", "3,5,4,4", "2,6,4,4", "2,7,3,3", "4,4,4,4"])
def test_v_rings_longer_than_the_hand_over_ring(ctx, oracle_mod, monkeypatch, ring):
    """More V slots than hand-over barriers (they fit at head_dim 64): the slot of the last tile, whose
    rows beyond kv_len are zeroed, was used by a tile whose barrier may be two phases on."""
    monkeypatch.setenv("LVSPEC_TC_RING", ring)
    kv_len = [128 * n + 63 for n in (37, 30, 9, 12)]
    case = _junk_beyond(A._case(78, 4, 8, 10, 2, 64, 128 * 38, kv_len, [[130, 1100]] * 4), kv_len)
    A._check(ctx, oracle_mod, case, n_split=1, kernel=2)
    A._check(ctx, oracle_mod, case, n_split=2, kernel=2)


@pytest.mark.parametrize("branch", [(1, 3), (2, 5), (5, 2), (13, 1)])
def test_draft_ranges(ctx, oracle_mod, branch):
    """Which draft slots a column sees, as a range of columns per slot: trees of several
    shapes, their slots across a tile boundary."""
    import test_gpu_tree as TR
    from gpu_util import assert_attention_close
    n_branches, length = branch
    kv_len = [640, 128 * 3 + length]
    case = TR._case(51, 2, n_branches, length, 8, 2, 128, kv_len, [[3, 500], [0, 300]])
    ref_out, ref_mass = oracle_mod.verify_attention(*case, branch_len=length)
    for n_split in (1, 3):
        out, mass, _ = TR._run_tree(ctx, case, n_branches, 2, n_split)
        assert_attention_close(out, mass, ref_out, ref_mass)
