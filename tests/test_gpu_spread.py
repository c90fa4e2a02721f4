"""GPU: appends whose grids sit at the edges of the rule that spreads early blocks over the SMs.

Each append stands right behind an attention call over its stream, without a synchronisation, on grids of one block an
SM more or less, of the largest even share that is spread and one block beyond, and of a full chip.  Reference:
plain torch in 64 bits, one rounding to bf16."""
import pytest
import torch

from paper_2509_22622_b200 import binding as B

pytestmark = pytest.mark.gpu

HEADS, DIM = 1, 64
SMS = 148
# tokens per block: 32 (rotation and append of one head of 64), 4 (with the norm)
EDGES = [(kind, tokens) for kind, per_block, full in (("plain", 32, 3), ("e4m3", 32, 2), ("norm", 4, 9))
         for blocks in sorted({1, SMS, SMS + 1, min(4, full - 1) * SMS, min(4, full - 1) * SMS + 1, full * SMS + 1})
         for tokens in (blocks * per_block,)]


@pytest.mark.parametrize("kind,tokens", EDGES)
def test_appends_at_the_edges_of_the_spread(kind, tokens):
    gen = torch.Generator(device="cuda").manual_seed(tokens)
    fmt = dict(kv_format=B.LL_KV_E4M3) if kind == "e4m3" else {}
    cache = B.Cache(1, HEADS, DIM, tokens, 1, 1, 2, **fmt)
    if fmt:
        cache.set_kv_scales(0, [0.015625] * HEADS, [0.015625] * HEADS)
    q, k, v = (torch.randn(tokens, HEADS, DIM, device="cuda", generator=gen).to(torch.bfloat16) for _ in range(3))
    gain = torch.rand(HEADS * DIM, device="cuda", generator=gen) + 0.5
    q_out, out = (torch.full_like(q, float("nan")) for _ in range(2))
    cache.rope_append_kv(0, q, v, k, 0, 1, tokens, 10000.0, q_out)
    torch.cuda.synchronize()
    for frame in (1, 1, 1):                          # a new frame, then over it again, each behind the attention before
        cache.sink_window_attn(0, q_out, 0 if frame > cache.state()["end"] - 1 else frame, out)
        if kind == "norm":
            cache.norm_rope_append_kv(0, q, k, v, gain, gain, 1e-6, frame, 1, tokens, 10000.0, q_out)
        else:
            cache.rope_append_kv(0, q, k, v, frame, 1, tokens, 10000.0, q_out)
    cache.check_device()

    n_h = DIM // 6
    n_t = DIM // 2 - 2 * n_h
    at = torch.arange(tokens, device="cuda", dtype=torch.float64)
    angle = torch.cat([a[:, None] * 10000.0 ** (-torch.arange(m, device="cuda", dtype=torch.float64) / m)
                       for a, m in ((torch.ones_like(at), n_t), (torch.zeros_like(at), n_h), (at, n_h))], 1)[:, None]

    def turned(x):
        x = x.double()
        if kind == "norm":
            x = x * (x.flatten(1).square().mean(1) + 1e-6).rsqrt()[:, None, None] * gain.double().reshape(HEADS, DIM)
        a, b, cos, sin = x[..., 0::2], x[..., 1::2], angle.cos(), angle.sin()
        return torch.stack([a * cos - b * sin, a * sin + b * cos], -1).flatten(-2)

    stored = [cache.kv_view(0, i)[:, tokens:2 * tokens].transpose(0, 1) for i in range(2)]
    # one rounding to bf16 (2^-8 of the element) on an fp32 rotation (1e-5 of values of a few units)
    assert ((q_out.double() - turned(q)).abs() <= 2.0 ** -8 * turned(q).abs() + 1e-5).all()
    if fmt:
        codes = [s.contiguous().view(torch.float8_e4m3fn).double() * 0.015625 for s in stored]
        # four significant bits (2^-4 of the element), the smallest step 2^-10 of the scale's 2^-6
        for got, want in zip(codes, (turned(k), v.double())):
            assert ((got - want).abs() <= 2.0 ** -4 * want.abs() + 2.0 ** -15).all()
    else:
        assert ((stored[0].double() - turned(k)).abs() <= 2.0 ** -8 * turned(k).abs() + 1e-5).all()
        assert torch.equal(stored[1], v)
    cache.close()
