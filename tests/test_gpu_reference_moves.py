"""GPU parity where the softmax references have to move.

The attention kernel computes a 64-key piece against the reference maxima of the
keys before it and moves the references of a warp's rows when the sum of the 16
weights that a thread holds of a row reaches 128: a single score seven octaves above
its reference, or sixteen of them three octaves above.  Random activations seldom do
that, so the scores here are made to: one feature of the keys climbs by a chosen
number of octaves at chosen keys (in the first and in the second piece of a step, at
the first key of a step, at the last), and the queries follow it with different
signs and strengths, so that within one warp some rows move and others do not."""
import numpy as np
import pytest
import torch

from paper_2509_22622_b200 import binding as B

from gpu_util import f64

pytestmark = pytest.mark.gpu


def check_climb(head_dim, climb, n_q, seed, scale=1.0):
    heads, n_k = 3, len(climb)
    gen = torch.Generator().manual_seed(seed)
    q, k, v = (torch.randn(n, heads, head_dim, generator=gen) for n in (n_q, n_k, n_k))
    q *= scale
    # feature 0 adds strength * climb octaves to a score: strengths 1, 0.5, 0, -1 row by row
    strength = torch.tensor([1.0, 0.5, 0.0, -1.0]).repeat(n_q // 4 + 1)[:n_q]
    q[:, :, 0] = strength[:, None] * 8.0
    k[:, :, 0] = (climb * (head_dim ** 0.5) / 1.4426950408889634 / 8.0)[:, None]
    q, k, v = (t.to(torch.bfloat16).cuda() for t in (q, k, v))
    cache = B.Cache(1, heads, head_dim, 16, 1, 1, 1)
    out = torch.full_like(q, float("nan"))
    lse = torch.full((heads, n_q), float("nan"), device="cuda")
    cache.cross_attn(q, k, v, out, lse)
    cache.check_device()
    s = torch.einsum("qhd,khd->hqk", q.double(), k.double()) * head_dim ** -0.5
    w = s.softmax(-1)
    want = torch.einsum("hqk,khd->qhd", w, v.double()).cpu().numpy()
    summed = torch.einsum("hqk,khd->qhd", w, v.double().abs()).cpu().numpy()
    want_lse = s.logsumexp(-1).cpu().numpy()
    # rounding the weights to bf16 moves an output by up to 2^-8 of what it sums, rounding the output by 2^-8 of itself
    # (rows here hang on a few keys, so both are reached); 1e-3 for the rest
    got = f64(out)
    assert np.isfinite(got).all()
    assert (np.abs(got - want) <= 2.0 ** -8 * (summed + np.abs(want)) + 1e-3).all()
    # scores are fp32 sums: 2^-20 of the largest, and the weights' own error (7.5e-5 of a weight at head_dim 64)
    assert np.abs(lse.cpu().numpy() - want_lse).max() <= 2e-4 + 2.0 ** -20 * s.abs().max().item()
    cache.close()


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("octaves", [5.0, 8.0, 33.0, 120.0, 300.0])
@pytest.mark.parametrize("n_q,n_k", [(40, 400), (300, 129)])
def test_scores_that_climb(head_dim, octaves, n_q, n_k):
    climb = torch.zeros(n_k)
    for at in (3, 64, 70, 128, 191, 255, 256, 383, 399):
        if at < n_k:
            climb[at:] += octaves
    check_climb(head_dim, climb, n_q, int(octaves) * 1000 + n_k + head_dim)


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("octaves,single", [(6.5, True), (7.5, True), (2.75, False), (3.25, False)])
def test_scores_on_both_sides_of_the_limit(head_dim, octaves, single):
    """One key a piece up by just under and just over seven octaves; all keys of a piece up by just under and just over three,
    so that no weight but their sum comes near the limit.  The other features only blur this: they are small here."""
    climb = torch.zeros(520)
    if single:
        climb[torch.tensor([70, 133, 200, 260, 390, 519])] = octaves
    else:
        climb[64:128] = octaves
        climb[256:320] = octaves
        climb[448:] = octaves
    check_climb(head_dim, climb, 40, int(4 * octaves) + head_dim, scale=0.05)
