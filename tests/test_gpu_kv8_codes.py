"""GPU: the codes of the 8-bit cache, byte for byte.

Codes are the E4M3 rounding (to nearest even, saturating) of the correctly rounded fp32 quotient by the head's scale.  The
kernel takes the quotient from a reciprocal for ordinary scales and divides for extreme ones; both are
compared with torch's division on every kind of value: zeros of both signs, values that underflow, that sit on
rounding boundaries, that saturate, infinities and NaN."""
import pytest
import torch

from paper_2509_22622_b200 import binding as B

pytestmark = pytest.mark.gpu

SCALES = [6.0 / 448.0, 1.0, 3.0, 0.7310586, 2.0 ** -60, 2.0 ** 60, 1.1 * 2.0 ** -61, 1e30, 1e-30]


@pytest.mark.parametrize("dim,gh,gw", [(64, 5, 7), (128, 16, 33)])
def test_codes_are_the_rounded_quotients(dim, gh, gw):
    heads, n = len(SCALES), gh * gw
    gen = torch.Generator(device="cuda").manual_seed(dim)
    cache = B.Cache(1, heads, dim, n, 1, 1, 2, kv_format=B.LL_KV_E4M3)
    cache.set_kv_scales(0, SCALES, SCALES)
    scale = torch.tensor(SCALES, device="cuda", dtype=torch.float32)[None, :, None]
    # values spread over the codes' range and beyond on both sides, times the head's scale
    spread = torch.exp2(torch.randint(-14, 12, (n, heads, dim), device="cuda", generator=gen).float())
    v = (torch.randn(n, heads, dim, device="cuda", generator=gen) * spread * scale).to(torch.bfloat16)
    k = (torch.randn(n, heads, dim, device="cuda", generator=gen) * spread * scale).to(torch.bfloat16)
    special = torch.tensor([0.0, -0.0, float("inf"), -float("inf"), float("nan"), 1e-38, -1e-38, 3e38], device="cuda").to(torch.bfloat16)
    v[0, :, :8] = special
    # quotients on and next to rounding boundaries of the codes (exact products where the scale is a power of two)
    v[1, :, :16] = ((torch.arange(16, device="cuda") + 0.5) / 8 * scale[0]).to(torch.bfloat16)
    cache.rope_append_kv(0, None, k, v, 0, gh, gw, 10000.0)
    cache.check_device()
    got = cache.kv_view(0, 1)[:, :n].transpose(0, 1)
    want = (v.float() / scale).clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8)
    nan = (v.float() / scale).isnan()
    assert torch.equal(got[~nan], want[~nan])
    assert ((got[nan] & 0x7f) == 0x7f).all()
    # token 0 of frame 0 is turned by angle 0: its k codes up to the sign of a zero
    got_k = cache.kv_view(0, 0)[:, 0]
    want_k = (k[0].float() / scale[0]).clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8)
    assert torch.equal(got_k & 0x7f, want_k & 0x7f)
    cache.close()
