"""GPU parity where an attention launch goes out by 128-row tiles: a tile alone, pairs, a pair and one left over, CTAs whose
tiles lie in two heads or in two groups (streams, chunks of a clip), one row in a head's last tile; bf16 and 8-bit caches, a
factor per query row, a recache."""
import numpy as np
import pytest
import torch

from paper_2509_22622_b200 import binding as B
from paper_2509_22622_b200 import synth

from gpu_util import bits, check_attn, dev, f64, new_cache

pytestmark = pytest.mark.gpu

F64 = synth.bf16_bits_to_f64


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("heads,P,chunks,by_tiles", [
    (12, 130, 3, True),          # 24 tiles on 24 SMs, two rows in every second
    (8, 385, 2, True),           # 32 tiles, one row in the last of a head
    (40, 769, 1, True),          # 280 tiles on 148 SMs: one or two each, some in two heads
    (40, 897, 1, True),          # 320 tiles, two or three each: pairs and a tile alone
    (24, 1210, 1, False),        # 240 tiles, by columns
    (16, 129, 1, True),          # two tiles a head, the second with one row
])
def test_decode_by_tiles(heads, P, chunks, by_tiles, D):
    wl = synth.Workload("tiles_%d_%d" % (heads, P), 1, heads, D, 1, P, 1, 0, 3, n_chunks=chunks, seed=700 + P)
    cache = new_cache(wl)
    for chunk in range(chunks):
        q, k, v = synth.chunk_qkv(wl, chunk)
        dq = dev(q)
        q_out = torch.empty_like(dq)
        cache.rope_append_kv(0, dq, dev(k), dev(v), chunk, 1, P, wl.rope_theta, q_out)
    assert (B.ll_debug_attn_tiles(cache.h)[0] > 0) == by_tiles
    out = torch.full_like(dq, float("nan"))
    lse = torch.full((heads, P), float("nan"), device="cuda")
    cache.sink_window_attn(0, q_out, chunks - 1, out, lse)
    cache.check_device()
    kc, vc = (cache.kv_view(0, i)[:, :chunks * P].double() for i in (0, 1))
    s = torch.einsum("qhd,hkd->hqk", q_out.double(), kc) * D ** -0.5
    want = torch.einsum("hqk,hkd->qhd", s.softmax(-1), vc).cpu().numpy()
    check_attn(f64(out), want)
    assert (lse.double() - s.logsumexp(-1)).abs().max().item() <= 1e-3
    again = torch.empty_like(out)
    cache.sink_window_attn(0, q_out, chunks - 1, again)
    assert np.array_equal(bits(again), bits(out))
    cache.close()


def keys_values(cache, rows, scales=None):
    """The first cache rows as fp64, codes times their head's scale."""
    kv = [cache.kv_view(0, i)[:, :rows] for i in (0, 1)]
    if scales is None:
        return [x.double() for x in kv]
    return [x.contiguous().view(torch.float8_e4m3fn).double() * torch.tensor(sc, device="cuda", dtype=torch.float64)[:, None, None]
            for x, sc in zip(kv, scales)]


def attend(q, kc, vc):
    s = torch.einsum("qhd,hkd->hqk", q.double(), kc) * q.shape[-1] ** -0.5
    return torch.einsum("hqk,hkd->qhd", s.softmax(-1), vc), s.logsumexp(-1)


def fill(cache, wl, chunks, stream=0):
    """Appends `chunks` chunks; the last one's rotated q."""
    for chunk in range(chunks):
        q, k, v = synth.chunk_qkv(wl, chunk, stream=stream)
        dq = dev(q)
        q_out = torch.empty_like(dq)
        cache.rope_append_kv(0, dq, dev(k), dev(v), chunk, wl.grid_h, wl.grid_w, wl.rope_theta, q_out)
    return q_out


@pytest.mark.parametrize("D", [64, 128])
def test_streams_of_equal_length_by_tiles(D):
    """Six streams, every other one with an 8-bit cache: two CTAs have tiles of two streams."""
    heads, P, chunks = 13, 300, 2
    streams = []
    for i in range(6):
        wl = synth.Workload("tiles_batched_%d" % D, 1, heads, D, 1, P, 1, 0, 3, n_chunks=chunks, seed=720 + i)
        cache = B.Cache(*wl.cache_args, kv_format=B.LL_KV_E4M3 if i % 2 else 0)
        scales = None
        if i % 2:
            scales = [[6.0 / 448 * (1 + 0.1 * h) * f for h in range(heads)] for f in (1.0, 0.8)]
            cache.set_kv_scales(0, *scales)
        q_out = fill(cache, wl, chunks, stream=i)
        out = torch.full_like(q_out, float("nan"))
        lse = torch.full((heads, P), float("nan"), device="cuda")
        streams.append((cache, 0, q_out, chunks - 1, out, lse, scales))
    plan = B.ll_debug_attn_plan_batched([(s[0].h, 0) for s in streams], 148)
    assert (plan.tile_ctas, plan.tiles_each, plan.tiles_extra, plan.row_tiles[0]) == (148, 1, 86, 3)
    B.Cache.sink_window_attn_batched([s[:6] for s in streams])
    for cache, _, q_out, _, out, lse, scales in streams:
        cache.check_device()
        want, want_lse = attend(q_out, *keys_values(cache, chunks * P, scales))
        check_attn(f64(out), want.cpu().numpy())
        assert (lse.double() - want_lse).abs().max().item() <= 1e-3
        cache.close()


@pytest.mark.parametrize("D", [64, 128])
def test_clip_chunks_of_equal_length_by_tiles(D):
    heads, P, n, window = 13, 300, 6, 2
    wl = synth.Workload("tiles_clip_%d" % D, 1, heads, D, 1, P, 1, 0, 12, n_chunks=0, seed=730)
    cache = new_cache(wl)
    fill(cache, wl, 1)
    q, k, v = synth.chunk_qkv(wl, 100, n_frames=n)
    dq = dev(q)
    q_out, out = torch.empty_like(dq), torch.full_like(dq, float("nan"))
    lse = torch.full((heads, n * P), float("nan"), device="cuda")
    cache.clip_append_attn(0, dq, dev(k), dev(v), 1, n, window, 1, P, wl.rope_theta, q_out, out, lse)
    plan = B.ll_debug_attn_plan_clip(cache.h, n, window, sm_count=148)
    assert (plan.tile_ctas, plan.tiles_each, plan.tiles_extra, plan.n_groups) == (148, 1, 86, n)
    cache.check_device()
    kc, vc = keys_values(cache, (n + 1) * P)
    for g in range(n):
        rows, seen = slice(g * P, (g + 1) * P), slice(g * P, (g + 2) * P)    # the chunk itself and the one before it
        want, want_lse = attend(q_out[rows], kc[:, seen], vc[:, seen])
        check_attn(f64(out[rows]), want.cpu().numpy())
        assert (lse[:, rows].double() - want_lse).abs().max().item() <= 1e-3
    cache.close()


@pytest.mark.parametrize("D", [64, 128])
def test_row_factors_and_recache_by_tiles(D):
    heads, P = 12, 390
    wl = synth.Workload("tiles_scaled_%d" % D, 1, heads, D, 1, P, 1, 0, 1, n_chunks=1, seed=740)
    cache = new_cache(wl)
    q_out = fill(cache, wl, 1)
    factor = 0.5 + torch.rand(P, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    assert B.ll_debug_attn_plan(cache.h, sm_count=148).tile_ctas == B.ll_debug_attn_plan(cache.h, recache=True, sm_count=148).tile_ctas == 48
    out = torch.full_like(q_out, float("nan"))
    B.ll_sink_window_attn_scaled(cache.h, 0, q_out, factor, 0, 1, out)
    cache.check_device()
    want, _ = attend(q_out.double() * factor.double()[:, None, None], *keys_values(cache, P))
    check_attn(f64(out), want.cpu().numpy())
    rq, rk, rv = synth.chunk_qkv(wl, 1, pass_id=synth.RECACHE_PASS)
    rq_out, out = torch.empty_like(q_out), torch.full_like(q_out, float("nan"))
    cache.recache(0, dev(rq), dev(rk), dev(rv), 1, 1, P, wl.rope_theta, rq_out, out)
    cache.check_device()
    want, _ = attend(rq_out, *keys_values(cache, P))
    check_attn(f64(out), want.cpu().numpy())
    cache.close()
