"""GPU parity of the fused projection at the edges of its tiles.

A pair of CTAs works on 256 tokens x 256, 192 or 128 features.  The shapes here sit at the edges:
one token, a last tile of one row, one CTA of the pair without rows, every tile width at both head sizes, more tiles than
pairs (accumulator buffers reused), K blocks with a tail, rows of one and of several sweeps of the norm's second kernel.  What
a shape is there for - tile width, tiles of the busiest pair - is asked of the library.  Reference: plain torch in 64 bits."""
import pytest
import torch

from paper_2509_22622_b200 import binding as B

pytestmark = pytest.mark.gpu

# heads, head_dim, grid_h, grid_w, d_model; tile width, tiles of the busiest pair
SHAPES = [
    (2, 128, 1, 1, 64, 128, 1),         # one token, one K block
    (4, 64, 1, 129, 72, 128, 1),        # the second CTA holds one row; K tail of 8
    (3, 64, 1, 255, 1544, 192, 1),      # last row missing
    (3, 128, 1, 257, 128, 128, 1),      # a tile of one row
    (2, 128, 79, 80, 136, 128, 3),      # 25 tiles of 256 tokens
    (12, 128, 10, 52, 384, 192, 1),
    (24, 64, 30, 156, 136, 256, 5),     # the widest tiles at head_dim 64, both accumulator buffers used again
    (12, 128, 30, 156, 72, 256, 5),
    (9, 64, 1, 4100, 72, 192, 3),       # both accumulator buffers used again at width 192
    (3, 128, 100, 124, 64, 192, 4),
    (12, 64, 79, 80, 64, 128, 7),
    (40, 128, 1, 130, 200, 256, 1),     # 5120 features: four sweeps of the norm's second kernel
    (64, 128, 1, 40, 64, 128, 3),       # 8192, the most that is accepted
]


def turn(x, cos, sin):
    a, b = x[..., 0::2], x[..., 1::2]
    return torch.stack([a * cos - b * sin, a * sin + b * cos], -1).flatten(-2)


@pytest.mark.parametrize("with_norm", [False, True], ids=["plain", "norm"])
@pytest.mark.parametrize("heads,dim,gh,gw,d_model,tile_n,per_pair", SHAPES)
def test_tile_edges(heads, dim, gh, gw, d_model, tile_n, per_pair, with_norm):
    n, width = gh * gw, heads * dim
    assert B.ll_debug_qkv_tiles(n, width, 148) == (tile_n, per_pair)
    gen = torch.Generator(device="cuda").manual_seed(n + d_model)
    x = torch.randn(n, d_model, device="cuda", generator=gen).to(torch.bfloat16)
    w = (torch.randn(3 * width, d_model, device="cuda", generator=gen) * d_model ** -0.5).to(torch.bfloat16)
    bias = torch.randn(3 * width, device="cuda", generator=gen) * 0.1
    gq, gk = (1 + 0.1 * torch.randn(width, device="cuda", generator=gen) for _ in range(2))
    cache = B.Cache(1, heads, dim, n, 1, 1, 2)
    q_out = torch.full((n, heads, dim), float("nan"), device="cuda", dtype=torch.bfloat16)
    scale = torch.full((n,), float("nan"), device="cuda")
    ws = torch.empty(B.ll_qkv_proj_workspace_bytes(cache.h) + 256, dtype=torch.uint8, device="cuda")
    ws = ws[(-ws.data_ptr()) % 256:]
    for frame in range(2):                       # the sink slot, then a ring slot
        B.ll_qkv_proj_append(cache.h, 0, x, w, bias, gq if with_norm else None, gk if with_norm else None, 1e-6, frame, 1,
                             gh, gw, 10000.0, q_out, scale if with_norm else None, ws if with_norm else None)
    cache.check_device()
    y = (x.double() @ w.double().T + bias.double()).reshape(n, 3, heads, dim)
    q, k, v = y[:, 0], y[:, 1], y[:, 2]
    if with_norm:
        rq, rk = ((t.flatten(1).square().mean(1) + 1e-6).rsqrt() for t in (q, k))
        assert ((scale.double() / rq - 1).abs() <= 1e-5).all()
        q, k = q * gq.double().reshape(heads, dim), k * gk.double().reshape(heads, dim) * rk[:, None, None]
    n_h = dim // 6
    n_t = dim // 2 - 2 * n_h
    at = torch.arange(n, device="cuda")
    angle = torch.cat([a.double()[:, None] * 10000.0 ** (-torch.arange(m, device="cuda", dtype=torch.float64) / m)
                       for a, m in ((torch.ones_like(at), n_t), (at // gw, n_h), (at % gw, n_h))], 1)[:, None]
    stored = [cache.kv_view(0, i)[:, n:2 * n].transpose(0, 1) for i in range(2)]
    for got, want in ((q_out, turn(q, angle.cos(), angle.sin())), (stored[0], turn(k, angle.cos(), angle.sin())), (stored[1], v)):
        # one rounding to bf16 (2^-8 of the element) on fp32 sums of d_model products (1e-4 covers their order)
        assert ((got.double() - want).abs() <= 2.0 ** -8 * want.abs() + 1e-4).all()
    cache.close()


@pytest.mark.parametrize("heads,dim,tokens,d_model,tile_n", [(2, 128, 1, 64, 128), (3, 64, 255, 1544, 192), (12, 128, 4680, 136, 256)])
def test_behind_a_recorded_timeout(heads, dim, tokens, d_model, tile_n):
    """Projections behind a time-out that nobody has read yet write nothing and end at once, pairs and all; the same call works
    when it has been read."""
    width = heads * dim
    assert B.ll_debug_qkv_tiles(tokens, width, 148)[0] == tile_n
    gen = torch.Generator(device="cuda").manual_seed(tokens)
    x = torch.randn(tokens, d_model, device="cuda", generator=gen).to(torch.bfloat16)
    w = torch.randn(3 * width, d_model, device="cuda", generator=gen).to(torch.bfloat16)
    cache = B.Cache(1, heads, dim, tokens, 1, 1, 2)
    q_out = torch.empty(tokens, heads, dim, device="cuda", dtype=torch.bfloat16)

    def project():
        B.ll_qkv_proj_append(cache.h, 0, x, w, None, None, None, 1e-6, 0, 1, 1, tokens, 10000.0, q_out)

    def rows():
        return [q_out] + [cache.kv_view(0, i)[:, :tokens] for i in range(2)]

    project()
    cache.check_device()
    want = [t.clone() for t in rows()]
    for t in rows():
        t.fill_(7.0)
    begin, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    B.ll_debug_wait_timeout(cache.h, 20)
    begin.record()
    for _ in range(10):
        project()
    end.record()
    torch.cuda.synchronize()
    assert all(bool((t == 7.0).all()) for t in rows())
    assert begin.elapsed_time(end) < 40.0                # 0.2 ms each, in which copies under way land
    with pytest.raises(B.LLError) as e:
        cache.check_device()
    assert e.value.code == B.LL_ERR_DEVICE_TIMEOUT
    project()
    cache.check_device()
    assert all(torch.equal(t, a) for t, a in zip(rows(), want))
    cache.close()
