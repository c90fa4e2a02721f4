"""GPU: the norm's append on rows and gains far from 1.

The factor of a row brings its elements to the order of 1 before the gain multiplies them, so a row of large (small)
elements with large (small) gains has results in range although element times gain is not."""
import pytest
import torch

from paper_2509_22622_b200 import binding as B

pytestmark = pytest.mark.gpu

GH, GW, THETA = 2, 5, 10000.0


@pytest.mark.parametrize("heads,dim", [(2, 64), (12, 128), (40, 128)])     # rows kept in registers, and read again
@pytest.mark.parametrize("size,gain_size", [(1e15, 1e26), (1e-17, 1e-25), (1e17, 1e-30), (1.0, 1.0)])
def test_element_times_gain_out_of_range(heads, dim, size, gain_size):
    n, width = GH * GW, heads * dim
    gen = torch.Generator(device="cuda").manual_seed(heads)
    q, k, v = ((torch.randn(n, heads, dim, device="cuda", generator=gen) * size).to(torch.bfloat16) for _ in range(3))
    gq, gk = ((torch.rand(width, device="cuda", generator=gen) + 0.5) * gain_size for _ in range(2))
    cache = B.Cache(1, heads, dim, n, 1, 1, 2)
    q_out = torch.full_like(q, float("nan"))
    cache.norm_rope_append_kv(0, q, k, v, gq, gk, 0.0, 0, GH, GW, THETA, q_out)
    cache.check_device()
    n_h = dim // 6
    n_t = dim // 2 - 2 * n_h
    at = torch.arange(n, device="cuda")
    angle = torch.cat([a.double()[:, None] * THETA ** (-torch.arange(m, device="cuda", dtype=torch.float64) / m)
                       for a, m in ((torch.zeros_like(at), n_t), (at // GW, n_h), (at % GW, n_h))], 1)[:, None]
    for got, x, g in ((q_out, q, gq), (cache.kv_view(0, 0)[:, :n].transpose(0, 1), k, gk)):
        x = x.double()
        x = x * x.flatten(1).square().mean(1).rsqrt()[:, None, None] * g.double().reshape(heads, dim)
        a, b, cos, sin = x[..., 0::2], x[..., 1::2], angle.cos(), angle.sin()
        want = torch.stack([a * cos - b * sin, a * sin + b * cos], -1).flatten(-2)
        # one rounding to bf16, and the fp32 factors' error relative to the length of the turned pair
        pair = (a * a + b * b).sqrt().repeat_interleave(2, -1)
        assert ((got.double() - want).abs() <= 2.0 ** -8 * want.abs() + 8e-6 * pair).all()
    assert torch.equal(cache.kv_view(0, 1)[:, :n].transpose(0, 1), v)
    cache.close()


@pytest.mark.parametrize("heads,dim", [(2, 64), (40, 128)])
def test_a_row_whose_squares_overflow_gives_zeros(heads, dim):
    """The sum of squares is taken in fp32: it is infinite here and the factor zero."""
    n = GH * GW
    x = torch.full((n, heads, dim), 3e38, device="cuda", dtype=torch.bfloat16)
    gain = torch.full((heads * dim,), 2.0, device="cuda")
    cache = B.Cache(1, heads, dim, n, 1, 1, 2)
    q_out = torch.full_like(x, float("nan"))
    cache.norm_rope_append_kv(0, x, x, x, gain, gain, 1e-6, 0, GH, GW, THETA, q_out)
    cache.check_device()
    assert (q_out == 0).all() and (cache.kv_view(0, 0)[:, :n] == 0).all()
    cache.close()
