"""GPU parity of columns whose keys are split into many parts.

Parts are merged all at once up to four (two at head_dim 64), one by one beyond.  Streams of different lengths
in one launch give levelled shares, so their columns come in differing numbers of parts; the plan says in how many.
Reference: plain torch in 64 bits on the stored rows."""
import pytest
import torch

from paper_2509_22622_b200 import binding as B

from gpu_util import check_attn, f64

pytestmark = pytest.mark.gpu


def parts_per_column(plan):
    cuts = plan.share_begin[:plan.n_shares + 1]
    counts = set()
    for g in range(plan.n_groups):
        for col in range(plan.heads * plan.tiles[g] - plan.wave_cols[g]):
            first = plan.step_begin[g] + col * plan.n_kt[g]
            counts.add(sum(lo < first + plan.n_kt[g] and hi > first for lo, hi in zip(cuts, cuts[1:])))
    return counts


# heads, tokens per frame, frames appended by each stream, part counts that must occur
@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("heads,p,streams,wanted", [(8, 300, (7, 3), {3, 4, 6, 7}), (2, 300, (7, 5, 2), {5, 12, 17}), (3, 256, (7, 2), {4, 14}),
                                                     (16, 520, (6, 3, 2), {2, 3})])
def test_columns_in_many_parts(heads, p, streams, wanted, head_dim):
    gen = torch.Generator(device="cuda").manual_seed(heads)
    items, want = [], []
    for n in streams:
        cache = B.Cache(1, heads, head_dim, p, 1, 1, 6)
        for f in range(n):
            q, k, v = (torch.randn(p, heads, head_dim, device="cuda", generator=gen).to(torch.bfloat16) for _ in range(3))
            q_out = torch.empty_like(q)
            cache.rope_append_kv(0, q, k, v, f, 1, p, 10000.0, q_out)
        out = torch.full_like(q, float("nan"))
        lse = torch.full((heads, p), float("nan"), device="cuda")
        items.append((cache, 0, q_out, n - 1, out, lse))
        kc, vc = (cache.kv_view(0, i)[:, :n * p].double() for i in range(2))
        s = torch.einsum("qhd,hkd->hqk", q_out.double(), kc) * head_dim ** -0.5
        want.append((torch.einsum("hqk,hkd->qhd", s.softmax(-1), vc), s.logsumexp(-1)))
    plan = B.ll_debug_attn_plan_batched([(c.h, 0) for c, *_ in items], sm_count=148)
    assert wanted <= parts_per_column(plan), parts_per_column(plan)
    for _ in range(2):                               # the second launch finds the first one's scratch and counters
        B.Cache.sink_window_attn_batched(items)
    for (cache, _, _, _, out, lse), (ref, ref_lse) in zip(items, want):
        cache.check_device()
        check_attn(f64(out), ref.cpu().numpy())
        assert (lse.double() - ref_lse).abs().max().item() <= 1e-4
        cache.close()
