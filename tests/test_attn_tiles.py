"""CPU-only: the division of an attention launch by 128-row tiles.

The rule a CTA follows is written out again in Python; every tile of every head is taken exactly once, two at a time only
inside a head, and no CTA ends later than with the division into columns that is used otherwise (a tile alone counted
as 0.7 of a column, 0.76 at head_dim 64)."""
import pytest
from hypothesis import given, settings, strategies as st

from paper_2509_22622_b200 import binding as B

from test_attn_plan import cta_work, make_cache

ALONE = {64: 0.76, 128: 0.7}


def segments(plan):
    """Per CTA its (group, head, first tile of the head, tiles); tiles numbered head after head, group after group."""
    at = [(g, h, t) for g in range(plan.n_groups) for h in range(plan.heads) for t in range(plan.row_tiles[g])]
    for i in range(plan.tile_ctas):
        u = i * plan.tiles_each + min(i, plan.tiles_extra)
        end = u + plan.tiles_each + (i < plan.tiles_extra)
        out = []
        while u < end:
            g, h, t = at[u]
            n = min(2, end - u, plan.row_tiles[g] - t)
            out.append((g, h, t, n))
            u += n
        yield out


def check_tiles(plan, rows, dim, sms):
    """What must hold of a plan whose groups have `rows` queries; its CTAs' segments if it goes by tiles."""
    assert list(plan.row_tiles[:plan.n_groups]) == [(rows + 127) // 128] * plan.n_groups
    if not plan.tile_ctas:
        assert (plan.tiles_each, plan.tiles_extra) == (0, 0)
        return []
    segs = list(segments(plan))
    taken = [(g, h, t + k) for s in segs for g, h, t, n in s for k in range(n)]
    assert taken == [(g, h, t) for g in range(plan.n_groups) for h in range(plan.heads) for t in range(plan.row_tiles[g])]
    assert plan.tile_ctas <= sms
    n_kt = plan.n_kt[0]
    assert all(plan.n_kt[g] == n_kt for g in range(plan.n_groups))
    by_tiles = max(sum(1. if n == 2 else ALONE[dim] for _, _, _, n in s) for s in segs) * n_kt
    # what splitting adds to the steps of the busiest CTA: the trip through the scratch slots, the merge by four parts, and
    # a second segment where the parts are not equal
    split = 0.
    if plan.n_shares:
        equal = plan.n_waves == 0 and plan.n_ctas == plan.n_shares and plan.n_shares % plan.all_cols == 0
        parts = plan.n_shares // plan.all_cols
        held = [0, 148, 74, 45, 33, 26, 22, 15, 15][parts] if parts <= 8 else 0          # clusters, whose CTAs merge together
        together = plan.all_cols <= min(held, sms // max(parts, 1))
        split = 8. if not equal else (3.5 if parts == 2 else 4. if parts <= 4 else 5.) if together else 2.5 + 2.5 * ((parts + 3) // 4)
    by_columns = max(sum(k1 - k0 for _, _, k0, k1 in cta_work(plan, i)) for i in range(plan.n_ctas)) + split
    assert by_tiles < by_columns
    return segs


def check(heads, P, C, S, W, chunks, sms):
    """Whether the newest chunk goes out by tiles; if so, how."""
    h = make_cache(heads, P, C, S, W, chunks)
    tiles = B.ll_debug_attn_tiles(h, sm_count=sms)
    plan = B.ll_debug_attn_plan(h, sm_count=sms)
    B.ll_cache_destroy(h)
    assert tiles == (plan.tile_ctas, plan.tiles_each, plan.tiles_extra) and plan.n_groups == 1
    check_tiles(plan, C * P, 128, sms)
    return tiles


def test_where_the_line_lies():
    assert check(12, 130, 3, 3, 3, 1, 148) == (48, 1, 0)             # 24 columns of 4 steps, 48 tiles
    assert check(12, 493, 3, 3, 9, 6, 148)[0] == 0                   # 72 columns of 47 steps, in two parts each
    assert check(12, 1560, 3, 3, 9, 6, 148)[0] == 0                  # long columns: shares
    assert check(8, 550, 2, 0, 2, 1, 148) == (72, 1, 0)              # 40 columns of 9 steps: 72 tiles instead of parts
    assert check(40, 1000, 1, 0, 1, 1, 148) == (148, 2, 24)          # 160 columns of 8 steps, 12 of them shared otherwise
    assert check(2, 16, 1, 1, 2, 3, 148)[0] == 0                     # one tile a column already


@settings(max_examples=200, deadline=None, derandomize=True)
@given(heads=st.integers(1, 40), P=st.integers(1, 900), C=st.integers(1, 3), w_chunks=st.integers(1, 3), n_chunks=st.integers(1, 4),
       sms=st.sampled_from([1, 7, 148, 160]))
def test_every_tile_is_taken_once(heads, P, C, w_chunks, n_chunks, sms):
    check(heads, P, C, 0, w_chunks * C, n_chunks, sms)


def cache_of(heads, dim, P, W, n_chunks):
    h = B.ll_cache_create(1, heads, dim, P, 1, 0, W)
    B.ll_cache_set_dry_run(h, True)
    for chunk in range(n_chunks):
        B.ll_rope_append_kv(h, 0, None, None, None, chunk, 1, 1, P)
    return h


def crossing(segs):
    """CTAs whose tiles lie in two groups."""
    return sum(len({g for g, _, _, _ in s}) > 1 for s in segs)


def batched(heads, dim, P, n_chunks, streams, sms):
    handles = [cache_of(heads, dim, P, 4, n_chunks) for _ in range(streams)]
    plan = B.ll_debug_attn_plan_batched([(h, 0) for h in handles], sm_count=sms)
    for h in handles:
        B.ll_cache_destroy(h)
    assert plan.n_groups == streams
    return plan


def clip(heads, dim, P, clip_chunks, window, sms):
    h = cache_of(heads, dim, P, 12, window + clip_chunks - 1)
    plan = B.ll_debug_attn_plan_clip(h, clip_chunks, window, sm_count=sms)
    B.ll_cache_destroy(h)
    assert plan.n_groups == clip_chunks
    return plan


@pytest.mark.parametrize("dim", [64, 128])
def test_tiles_across_groups(dim):
    """156 columns of equally long groups of three tiles a head: two waves otherwise.  39 tiles a group, two a CTA:
    some lie in two groups."""
    for plan in (batched(13, dim, 300, 2, 6, 148), clip(13, dim, 300, 6, 2, 148)):
        segs = check_tiles(plan, 300, dim, 148)
        assert (plan.tile_ctas, plan.tiles_each, plan.tiles_extra) == (148, 1, 86) and crossing(segs) == 2


def test_groups_of_different_length_go_by_columns():
    handles = [cache_of(13, 128, 300, 4, n) for n in (1, 1, 1, 1, 1, 2)]
    plan = B.ll_debug_attn_plan_batched([(h, 0) for h in handles], sm_count=148)
    assert plan.tile_ctas == 0 and len({plan.n_kt[g] for g in range(6)}) == 2
    for h in handles:
        B.ll_cache_destroy(h)


def test_head_dim_64_has_a_line_of_its_own():
    """A pair and a tile alone are 1.7 of a column or 1.76, against 228 columns of 16 and of 24 steps in shares."""
    for n_k, by_tiles in ((2000, {64: 148, 128: 148}), (3072, {64: 0, 128: 148})):
        for dim in (64, 128):
            h = cache_of(12, dim, 16, 1, 1)
            plan = B.ll_debug_attn_plan_cross(h, 4680, n_k, sm_count=148)
            B.ll_cache_destroy(h)
            check_tiles(plan, 4680, dim, 148)
            assert plan.tile_ctas == by_tiles[dim]


def test_a_recache_of_one_chunk_and_cross_attention():
    h = cache_of(12, 128, 390, 1, 3)
    assert B.ll_debug_attn_plan(h, recache=True, sm_count=148).tile_ctas == 48
    plan = B.ll_debug_attn_plan_cross(h, 4680, 512, sm_count=148)
    assert (plan.tile_ctas, plan.tiles_each, plan.n_kt[0]) == (148, 3, 4)
    check_tiles(plan, 4680, 128, 148)
    assert B.ll_debug_attn_plan_cross(h, 1479, 47 * 128, sm_count=148).tile_ctas == 0
    for bad in ((0, 5), (5, 0)):
        with pytest.raises(B.LLError):
            B.ll_debug_attn_plan_cross(h, *bad)
    for bad in ((0, 1), (1, 0), (4, 1), (1, 2)):                     # frames, window: none, none, more than appended, more than the ring
        with pytest.raises(B.LLError):
            B.ll_debug_attn_plan_clip(h, *bad)
    B.ll_cache_destroy(h)


@settings(max_examples=100, deadline=None, derandomize=True)
@given(heads=st.integers(1, 40), dim=st.sampled_from([64, 128]), P=st.integers(1, 900), streams=st.integers(1, 8), n_chunks=st.integers(1, 4),
       is_clip=st.booleans(), sms=st.sampled_from([1, 7, 148, 160]))
def test_every_tile_of_several_groups_is_taken_once(heads, dim, P, streams, n_chunks, is_clip, sms):
    plan = clip(heads, dim, P, streams, min(n_chunks, 3), sms) if is_clip else batched(heads, dim, P, n_chunks, streams, sms)
    check_tiles(plan, P, dim, sms)
