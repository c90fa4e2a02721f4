"""Columns whose equal parts are held by the CTAs of a thread-block cluster, which merge them together.

Two to eight parts; one live row in a tile, two tiles, whole tiles; one query group or several; 8-bit caches and row factors.
Reference: plain torch in 64 bits on the stored rows, under the usual bar of the attention (tests/gpu_util.py)."""
import pytest
import torch

from paper_2509_22622_b200 import binding as B

# heads, head_dim, queries, keys, parts
SHAPES = [
    (12, 128, 1479, 5916, 2),               # 72 columns: two on 144 SMs
    (23, 64, 769, 47 * 128 - 1, 0),         # 92 columns: more than SMs for two parts
    (40, 128, 95, 9 * 128, 3),
    (2, 128, 300, 1500, 4),                 # the last column has one tile
    (24, 64, 200, 25 * 128 - 3, 5),
    (16, 128, 129, 22 * 128 - 127, 6),      # one row in the second tile, one key in the last
    (12, 128, 140, 14 * 128, 7),
    (12, 64, 1, 24 * 128, 8),               # one query
    (1, 64, 129, 5120, 8),
    (1, 128, 100, 10 * 128, 4),             # parts of two steps and of three
]


def handle(heads, dim):
    h = B.ll_cache_create(1, heads, dim, 16, 1, 1, 1)
    B.ll_cache_set_dry_run(h, True)
    return h


@pytest.mark.parametrize("heads,dim,n_q,n_k,parts", SHAPES)
def test_where_clusters_are_used(heads, dim, n_q, n_k, parts):
    h = handle(heads, dim)
    plan = B.ll_debug_attn_plan_cross(h, n_q, n_k, sm_count=148)
    B.ll_cache_destroy(h)
    assert plan.cluster_parts == parts
    if parts:
        cols = heads * ((n_q + 255) // 256)
        assert (plan.n_ctas, plan.n_shares, plan.n_waves, plan.tile_ctas) == (cols * parts, cols * parts, 0, 0)
        assert list(plan.share_of_cta[:plan.n_ctas]) == list(range(plan.n_ctas))
        # a CTA works its share out from its number alone
        n_kt = plan.n_kt[0]
        cuts = [col * n_kt + i * n_kt // parts for col in range(cols) for i in range(parts)] + [cols * n_kt]
        assert list(plan.share_begin[:plan.n_shares + 1]) == cuts


# what a device holds of each size; parts of SHAPES[0] (72 columns of 47 steps) and SHAPES[6] (12 columns of 14)
@pytest.mark.parametrize("held,parts", [([0, 148, 74, 45, 33, 26, 22, 15, 15], (2, 7)), ([0, 148, 71, 45, 33, 26, 22, 11, 15], (0, 8)),
                                        ([0, 148, 74, 45, 11, 26, 22, 0, 0], (2, 5)), ([0] * 9, (0, 0))])
def test_the_device_says_how_many_clusters(held, parts):
    """Clusters that would run one behind another are not planned with."""
    for (heads, dim, n_q, n_k, _), want in zip((SHAPES[0], SHAPES[6]), parts):
        h = handle(heads, dim)
        B.ll_debug_attn_clusters(h, held)
        assert B.ll_debug_attn_plan_cross(h, n_q, n_k).cluster_parts == want
        with pytest.raises(B.LLError):
            B.ll_debug_attn_clusters(h, [0, 0, 75] + [0] * 6)
        B.ll_cache_destroy(h)


@pytest.mark.gpu
@pytest.mark.parametrize("heads,dim,n_q,n_k,parts", [s for s in SHAPES if s[4]])
def test_without_clusters(heads, dim, n_q, n_k, parts):
    """The same launches on a device that holds none: the part that arrives last merges, or nothing is split."""
    from gpu_util import check_attn, f64
    gen = torch.Generator(device="cuda").manual_seed(n_q)
    q, k, v = (torch.randn(n, heads, dim, device="cuda", generator=gen).to(torch.bfloat16) for n in (n_q, n_k, n_k))
    cache = B.Cache(1, heads, dim, 16, 1, 1, 1)
    B.ll_debug_attn_clusters(cache.h, [0] * 9)
    plan = B.ll_debug_attn_plan_cross(cache.h, n_q, n_k)
    assert (plan.cluster_parts, plan.tile_ctas) == (0, 0) and plan.n_shares > plan.all_cols
    s = torch.einsum("qhd,khd->hqk", q.double(), k.double()) * dim ** -0.5
    want = torch.einsum("hqk,khd->qhd", s.softmax(-1), v.double()).cpu().numpy()
    for _ in range(2):
        out, lse = torch.full_like(q, float("nan")), torch.full((heads, n_q), float("nan"), device="cuda")
        cache.cross_attn(q, k, v, out, lse)
        cache.check_device()
        check_attn(f64(out), want)
        assert (lse.double() - s.logsumexp(-1)).abs().max().item() <= 1e-4
    cache.close()


@pytest.mark.gpu
@pytest.mark.parametrize("heads,dim,n_q,n_k,parts", [s for s in SHAPES if s[4]])
def test_cluster_parts(heads, dim, n_q, n_k, parts):
    from gpu_util import check_attn, f64, guarded
    gen = torch.Generator(device="cuda").manual_seed(n_q)
    q, k, v = (torch.randn(n, heads, dim, device="cuda", generator=gen).to(torch.bfloat16) for n in (n_q, n_k, n_k))
    cache = B.Cache(1, heads, dim, 16, 1, 1, 1)
    assert B.ll_debug_attn_plan_cross(cache.h, n_q, n_k).cluster_parts == parts
    outs = []
    for _ in range(3):                               # back to back: the next launch reuses the scratch of the one before
        out, guard = guarded((n_q, heads, dim), fill=float("nan"))
        lse = torch.full((heads, n_q), float("nan"), device="cuda")
        cache.cross_attn(q, k, v, out, lse)
        outs.append((out, guard, lse))
    cache.check_device()
    s = torch.einsum("qhd,khd->hqk", q.double(), k.double()) * dim ** -0.5
    want = torch.einsum("hqk,khd->qhd", s.softmax(-1), v.double()).cpu().numpy()
    for out, guard, lse in outs:
        guard()
        check_attn(f64(out), want)
        assert (lse.double() - s.logsumexp(-1)).abs().max().item() <= 1e-4
        assert torch.equal(out, outs[0][0]) and torch.equal(lse, outs[0][2])
    cache.close()


@pytest.mark.gpu
@pytest.mark.parametrize("dim", [64, 128])
def test_cluster_parts_of_a_cache(dim):
    """A stream's newest chunk over a wrapped ring: in bf16 with row factors, in 8 bits with per-head scales; two streams of one length."""
    from gpu_util import check_attn, f64
    heads, p, chunk, window, chunks = 8, 133, 3, 12, 6
    gen = torch.Generator(device="cuda").manual_seed(dim)

    def normal():
        return torch.randn(chunk * p, heads, dim, device="cuda", generator=gen).to(torch.bfloat16)

    def stream(kv_format):
        cache = B.Cache(1, heads, dim, p, chunk, chunk, window, kv_format=kv_format)
        scales = [[(1 + 0.1 * h) / 64 for h in range(heads)], [(2 - 0.1 * h) / 64 for h in range(heads)]]
        if kv_format:
            cache.set_kv_scales(0, *scales)
        for i in range(chunks):
            q_out = torch.empty_like(normal())
            cache.rope_append_kv(0, normal(), normal(), normal(), i * chunk, 1, p, 10000.0, q_out)
        k, v = (cache.kv_view(0, i) for i in range(2))
        if kv_format:
            k, v = (t.view(torch.float8_e4m3fn).double() * torch.tensor(s, dtype=torch.float32, device="cuda").double()[:, None, None]
                    for t, s in ((k, scales[0]), (v, scales[1])))
        return cache, q_out, k.double(), v.double()

    def want(q_out, k, v, factor):
        s = torch.einsum("qhd,hkd->hqk", q_out.double() * factor[:, None, None].double(), k) * dim ** -0.5
        return torch.einsum("hqk,hkd->qhd", s.softmax(-1), v).cpu().numpy()

    one = torch.ones(chunk * p, device="cuda")
    start = (chunks - 1) * chunk
    for kv_format, factor in ((B.LL_KV_BF16, None), (B.LL_KV_BF16, 0.5 + torch.rand(chunk * p, device="cuda", generator=gen)), (B.LL_KV_E4M3, None)):
        cache, q_out, k, v = stream(kv_format)
        assert B.ll_debug_attn_plan(cache.h).cluster_parts > 0
        out = torch.full_like(q_out, float("nan"))
        if factor is None:
            cache.sink_window_attn(0, q_out, start, out)
        else:
            B.ll_sink_window_attn_scaled(cache.h, 0, q_out, factor, start, chunk, out)
        cache.check_device()
        check_attn(f64(out), want(q_out, k, v, one if factor is None else factor))
        cache.close()
    streams = [stream(B.LL_KV_BF16) for _ in range(2)]
    assert B.ll_debug_attn_plan_batched([(c.h, 0) for c, *_ in streams]).cluster_parts > 0
    outs = [torch.full_like(q_out, float("nan")) for _, q_out, _, _ in streams]
    B.Cache.sink_window_attn_batched([(c, 0, q_out, start, out, None) for (c, q_out, _, _), out in zip(streams, outs)])
    for (cache, q_out, k, v), out in zip(streams, outs):
        cache.check_device()
        check_attn(f64(out), want(q_out, k, v, one))
        cache.close()


@pytest.mark.gpu
@pytest.mark.parametrize("dim", [64, 128])
def test_captured_cluster_parts(dim):
    """A launch of clusters between two others in a captured graph, replayed."""
    gen = torch.Generator(device="cuda").manual_seed(dim)
    q, k, v = (torch.randn(n, 8, dim, device="cuda", generator=gen).to(torch.bfloat16) for n in (450, 2300, 2300))
    cache = B.Cache(1, 8, dim, 16, 1, 1, 1)
    assert B.ll_debug_attn_plan_cross(cache.h, 450, 2300).cluster_parts > 0
    a, b, c = (torch.empty_like(q) for _ in range(3))
    want = []
    for src, dst in ((q, a), (a, b), (b, c)):
        cache.cross_attn(src, k, v, dst)
        torch.cuda.synchronize()
        want.append(dst.clone())
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        for src, dst in ((q, a), (a, b), (b, c)):
            cache.cross_attn(src, k, v, dst)
    for _ in range(3):
        for t in (a, b, c):
            t.fill_(float("nan"))
        graph.replay()
        assert all(torch.equal(t, w) for t, w in zip((a, b, c), want))
    cache.check_device()
    del graph
    cache.close()


@pytest.mark.gpu
def test_clusters_on_two_streams():
    """Launches of clusters of two handles side by side: each CTA waits only for those of its own cluster."""
    gen = torch.Generator(device="cuda").manual_seed(2)
    work = []
    for n_q, n_k in ((1479, 5916), (450, 2250)):
        q, k, v = (torch.randn(n, 12, 128, device="cuda", generator=gen).to(torch.bfloat16) for n in (n_q, n_k, n_k))
        cache = B.Cache(1, 12, 128, 16, 1, 1, 1)
        assert B.ll_debug_attn_plan_cross(cache.h, n_q, n_k).cluster_parts > 0
        want = torch.empty_like(q)
        cache.cross_attn(q, k, v, want)
        work.append((cache, q, k, v, torch.empty_like(q), want, torch.cuda.Stream()))
    torch.cuda.synchronize()
    for _ in range(20):
        for cache, q, k, v, out, _, stream in work:
            cache.cross_attn(q, k, v, out, stream=stream)
    torch.cuda.synchronize()
    for cache, _, _, _, out, want, stream in work:
        cache.check_device(stream)
        assert torch.equal(out, want)
        cache.close()


@pytest.mark.gpu
@pytest.mark.parametrize("heads,dim,n_q,n_k,parts", [s for s in SHAPES if s[4]])
def test_clusters_behind_a_recorded_timeout(heads, dim, n_q, n_k, parts):
    """Launches behind a time-out that nobody has read yet write nothing and end at once; the same call works when it has been read."""
    gen = torch.Generator(device="cuda").manual_seed(n_k)
    q, k, v = (torch.randn(n, heads, dim, device="cuda", generator=gen).to(torch.bfloat16) for n in (n_q, n_k, n_k))
    cache = B.Cache(1, heads, dim, 16, 1, 1, 1)
    assert B.ll_debug_attn_plan_cross(cache.h, n_q, n_k).cluster_parts == parts
    want = torch.empty_like(q)
    cache.cross_attn(q, k, v, want)
    cache.check_device()
    out = torch.full_like(q, 7.0)
    begin, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    B.ll_debug_wait_timeout(cache.h, 20)
    begin.record()
    for _ in range(10):
        cache.cross_attn(q, k, v, out)
    end.record()
    torch.cuda.synchronize()
    assert bool((out == 7.0).all())
    assert begin.elapsed_time(end) < 40.0                # 0.2 ms each, in which copies under way land
    with pytest.raises(B.LLError) as e:
        cache.check_device()
    assert e.value.code == B.LL_ERR_DEVICE_TIMEOUT
    cache.cross_attn(q, k, v, out)
    cache.check_device()
    assert torch.equal(out, want)
    cache.close()
