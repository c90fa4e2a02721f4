"""GPU parity of the append with the q/k norm where its kernel changes: rows and token counts on both sides of the line
between rows kept in registers, streamed through shared memory and read twice; fewer tokens than SMs, one more,
several rounds of tokens per warp; no q."""
import numpy as np
import pytest
import torch

from paper_2509_22622_b200 import binding as B
from paper_2509_22622_b200 import synth

from gpu_util import bits, dev, new_cache
from test_gpu_norm_append import EPS, F64, close_bits

pytestmark = pytest.mark.gpu


def case(name, heads, head_dim, grid_h, grid_w):
    return synth.Workload(name, 1, heads, head_dim, grid_h, grid_w, 1, 0, 1, n_chunks=1, seed=500 + heads + grid_w)


CASES = [
    case("4_heads", 4, 128, 5, 40),                # 64 vectors: registers
    case("5_heads", 5, 128, 1, 149),               # 80 vectors: streamed; one token more than SMs
    case("9_heads_of_64", 9, 64, 3, 5),            # 72 vectors, a ragged last round of lanes
    case("9_heads_of_64_rounds", 9, 64, 48, 148),  # registers from seven tokens an SM on
    case("9_heads_of_64_more", 9, 64, 71, 101),
    case("15_heads_of_64_rounds", 15, 64, 48, 148),    # the most tokens that are streamed
    case("12_heads", 12, 128, 17, 29),
    case("12_heads_registers", 12, 128, 37, 50),   # 13 tokens an SM
    case("12_heads_rounds", 12, 128, 42, 60),      # 18: two rounds of eleven warps
    case("16_heads_rounds", 16, 128, 45, 80),      # two reads without streaming
    case("17_heads", 17, 128, 16, 37),
    case("17_heads_more", 17, 128, 37, 65),        # read twice
    case("32_heads", 32, 128, 1, 1),               # four warps' buffers
    case("33_heads", 33, 128, 3, 7),               # fewer: read twice
]
STREAMED = {"5_heads", "9_heads_of_64", "15_heads_of_64_rounds", "12_heads", "12_heads_rounds", "16_heads_rounds", "17_heads", "32_heads"}


def run(wl, with_q=True):
    cache = new_cache(wl)
    q, k, v = synth.chunk_qkv(wl, 0)
    rng = np.random.default_rng(wl.seed)
    gq, gk = ((1.0 + 0.3 * rng.standard_normal((wl.heads, wl.head_dim))).astype(np.float32) for _ in range(2))
    dq = dev(q) if with_q else None
    q_out = torch.full_like(dq, float("nan")) if with_q else None
    cache.norm_rope_append_kv(0, dq, dev(k), dev(v), torch.from_numpy(gq).cuda() if with_q else None, torch.from_numpy(gk).cuda(), EPS, 0,
                              wl.grid_h, wl.grid_w, wl.rope_theta, q_out)
    cache.check_device()
    kc, vc = (bits(cache.kv_view(0, i)).transpose(1, 0, 2) for i in (0, 1))
    out = bits(q_out) if with_q else None
    cache.close()
    return (q, k, v, gq, gk), (out, kc, vc)


@pytest.mark.parametrize("wl", CASES, ids=lambda w: w.name)
def test_rows_and_rounds(oracle_mod, wl):
    assert B.ll_debug_norm_rows(wl.heads, wl.head_dim, wl.tokens_per_frame, sm_count=148) == (wl.name in STREAMED)
    (q, k, v, gq, gk), (out, kc, vc) = run(wl)
    for x, gain, got in ((q, gq, out), (k, gk, kc)):
        want = oracle_mod.rope(oracle_mod.rms_norm(F64(x), gain.astype(np.float64), EPS), 0, wl.grid_h, wl.grid_w, wl.rope_theta)
        close_bits(got, want)
    assert np.array_equal(vc, v)


@pytest.mark.parametrize("wl", [c for c in CASES if c.name in ("4_heads", "5_heads", "12_heads", "12_heads_registers", "16_heads_rounds", "33_heads")], ids=lambda w: w.name)
def test_without_q_the_cache_rows_are_the_same(wl):
    """k and v alone, by the same kernel or the other one: the bits of the call with q."""
    _, a = run(wl)
    _, b = run(wl, with_q=False)
    assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])
