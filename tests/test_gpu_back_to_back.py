"""GPU: calls enqueued back to back give the bits that the same calls give with a synchronisation after each.

Every kernel may start while the one in front of it is still running and waits for it before its first
access to memory.  The calls here hand results to one another (cache rows, rotated queries, outputs, scratch
slots and counters) from kernel to kernel, at sizes from a single block to split columns: one chain over a bf16 cache with
all entry points, one over an 8-bit cache, and one whose rotation tables are rewritten between the calls."""
import pytest
import torch

from paper_2509_22622_b200 import binding as B

pytestmark = pytest.mark.gpu


def pipeline(heads, dim, gh, gw, sync):
    gen = torch.Generator(device="cuda").manual_seed(7)
    p, width, theta = gh * gw, heads * dim, 10000.0

    def bf16(*shape):
        return torch.randn(*shape, device="cuda", generator=gen).to(torch.bfloat16)

    cache = B.Cache(1, heads, dim, p, 1, 1, 6)
    ws = torch.empty(B.ll_qkv_proj_workspace_bytes(cache.h) + 256, dtype=torch.uint8, device="cuda")
    ws = ws[(-ws.data_ptr()) % 256:]
    bws = torch.empty(B.ll_clip_backward_workspace_bytes(cache.h, 2) + 256, dtype=torch.uint8, device="cuda")
    bws = bws[(-bws.data_ptr()) % 256:]
    gain = torch.rand(width, device="cuda", generator=gen) + 0.5
    x, w = bf16(p, 256), bf16(3 * width, 256) * 0.06
    rounds = [[bf16(n * p, heads, dim) for n in (1, 1, 1, 2, 2, 2, 2, 6, 6, 6)] for _ in range(3)]
    one, two, six = (lambda n=n: torch.full((n * p, heads, dim), float("nan"), device="cuda", dtype=torch.bfloat16) for n in (1, 2, 6))
    kept = []
    torch.cuda.synchronize()

    def step(call, *args, **kw):
        call(*args, **kw)
        if sync:
            torch.cuda.synchronize()

    frame = 0
    for q, k, v, q2, k2, v2, g2, q6, k6, v6 in rounds:
        qo, o, o2, qc, oc, dq, dk, dv, qr, orc, oq, os, ox = one(), one(), one(), two(), two(), two(), two(), two(), six(), six(), one(), one(), one()
        lse, scale = torch.empty(heads, 2 * p, device="cuda"), torch.empty(p, device="cuda")
        step(cache.rope_append_kv, 0, q, k, v, frame, gh, gw, theta, qo)
        step(cache.sink_window_attn, 0, qo, frame, o)
        step(cache.norm_rope_append_kv, 0, o, k, o, gain, gain, 1e-6, frame, gh, gw, theta, qo)
        step(cache.sink_window_attn, 0, qo, frame, o2)
        step(B.ll_qkv_proj_append, cache.h, 0, x, w, None, gain, gain, 1e-6, frame, 1, gh, gw, theta, oq, scale, ws)
        step(B.ll_sink_window_attn_scaled, cache.h, 0, oq, scale, frame, 1, os)
        step(cache.cross_attn, os, o, o2, ox)
        frame += 1
        step(cache.clip_append_attn, 0, q2, k2, v2, frame, 2, 2, gh, gw, theta, qc, oc, lse)
        step(B.ll_clip_attn_backward, cache.h, 0, qc, oc, g2, lse, frame, 2, 2, gh, gw, theta, dq, dk, dv, bws)
        frame += 2
        n = min(6, frame - 1)
        step(cache.recache, 0, q6[:n * p], k6[:n * p], v6[:n * p], n, gh, gw, theta, qr[:n * p], orc[:n * p])
        kept += [qo, o, o2, oq, os, ox, qc, oc, lse, dq, dk, dv, qr[:n * p], orc[:n * p], scale]
    kept += [cache.kv_view(0, 0), cache.kv_view(0, 1)]
    cache.check_device()
    kept = [t.clone() for t in kept]
    cache.close()
    return kept


@pytest.mark.parametrize("heads,dim,gh,gw", [(4, 64, 2, 3), (2, 128, 12, 13), (12, 128, 16, 30)])
def test_calls_without_synchronisation(heads, dim, gh, gw):
    want = pipeline(heads, dim, gh, gw, True)
    for _ in range(3):
        got = pipeline(heads, dim, gh, gw, False)
        for i, (a, b) in enumerate(zip(got, want)):
            assert torch.equal(a, b), "tensor %d differs" % i
            assert not torch.isnan(a.float()).any(), "tensor %d holds unwritten rows" % i


def eight_bit(heads, dim, gh, gw, sync):
    """Append, attend, overwrite, attend over an 8-bit cache: append -> expansion -> attention, handing on cache rows,
    the expanded pair and outputs, and each next append writing over rows that the expansion in front of it reads."""
    gen = torch.Generator(device="cuda").manual_seed(11)
    p = gh * gw
    cache = B.Cache(1, heads, dim, p, 1, 1, 3, kv_format=B.LL_KV_E4M3)
    cache.set_kv_scales(0, [6.0 / 448.0] * heads, [6.0 / 448.0] * heads)
    rounds = [[torch.randn(p, heads, dim, device="cuda", generator=gen).to(torch.bfloat16) for _ in range(6)] for _ in range(6)]
    kept = []
    torch.cuda.synchronize()
    for frame, (q, k, v, k2, v2, v3) in enumerate(rounds):
        qo, o, o2, o3 = (torch.full_like(q, float("nan")) for _ in range(4))
        for kk, vv, out in ((k, v, o), (k2, v2, o2), (o2, v3, o3)):     # the last pass appends what attention just wrote
            for call in (lambda: cache.rope_append_kv(0, q, kk, vv, frame, gh, gw, 10000.0, qo),
                         lambda: cache.sink_window_attn(0, qo, frame, out)):
                call()
                if sync:
                    torch.cuda.synchronize()
        kept += [qo, o, o2, o3]
    kept += [cache.kv_view(0, 0), cache.kv_view(0, 1)]
    cache.check_device()
    kept = [t.clone() for t in kept]
    cache.close()
    return kept


def changing_tables(heads, dim, gh, gw, sync):
    """Calls that each need other rotation tables than the call before (another theta, the grid's sides swapped), so that
    the tables are rewritten between the kernels that read them."""
    gen = torch.Generator(device="cuda").manual_seed(13)
    p, width = gh * gw, heads * dim

    def bf16(*shape):
        return torch.randn(*shape, device="cuda", generator=gen).to(torch.bfloat16)

    cache = B.Cache(1, heads, dim, p, 1, 1, 4)
    bws = torch.empty(B.ll_clip_backward_workspace_bytes(cache.h, 2) + 256, dtype=torch.uint8, device="cuda")
    bws = bws[(-bws.data_ptr()) % 256:]
    gain = torch.rand(width, device="cuda", generator=gen) + 0.5
    x, w = bf16(p, 128), bf16(3 * width, 128) * 0.09
    q, k, v = (bf16(p, heads, dim) for _ in range(3))
    q2, k2, v2, g2 = (bf16(2 * p, heads, dim) for _ in range(4))
    turns = [(gh, gw, 10000.0), (gw, gh, 500.0), (gh, gw, 30.0), (gw, gh, 10000.0)]
    kept, at = [], 0
    torch.cuda.synchronize()

    def step(call):
        nonlocal at
        call(*turns[at % len(turns)])
        at += 1
        if sync:
            torch.cuda.synchronize()

    for frame in range(0, 12, 3):
        for passes in range(3):
            qo, qn, qp = (torch.full_like(q, float("nan")) for _ in range(3))
            step(lambda *t: cache.rope_append_kv(0, q, k, v, frame, *t, qo))
            step(lambda *t: cache.norm_rope_append_kv(0, q, k, v, gain, gain, 1e-6, frame, *t, qn))
            step(lambda *t: cache.rope_append_kv(0, q, k, v, frame, *t, qo))
            step(lambda *t: B.ll_qkv_proj_append(cache.h, 0, x, w, None, None, None, 0.0, frame, 1, *t, qp, None, None))
            step(lambda *t: cache.rope_append_kv(0, qo, qn, v, frame, *t, qn))
            kept.append((qo, qn, qp, cache.kv_view(0, 0).clone()))
        qc, oc, dq, dk, dv = (torch.full_like(q2, float("nan")) for _ in range(5))
        lse = torch.empty(heads, 2 * p, device="cuda")
        step(lambda *t: cache.clip_append_attn(0, q2, k2, v2, frame + 1, 2, 2, *t, qc, oc, lse))
        step(lambda *t: B.ll_clip_attn_backward(cache.h, 0, qc, oc, g2, lse, frame + 1, 2, 2, *t, dq, dk, dv, bws))
        kept.append((qc, oc, lse, dq, dk, dv))
    cache.check_device()
    kept = [t.clone() for group in kept for t in group]
    cache.close()
    return kept


@pytest.mark.parametrize("chain", [eight_bit, changing_tables])
@pytest.mark.parametrize("heads,dim,gh,gw", [(4, 64, 2, 3), (2, 128, 12, 13), (12, 128, 16, 30)])
def test_chains_without_synchronisation(chain, heads, dim, gh, gw):
    want = chain(heads, dim, gh, gw, True)
    for _ in range(3):
        got = chain(heads, dim, gh, gw, False)
        for i, (a, b) in enumerate(zip(got, want)):
            assert torch.equal(a, b), "tensor %d differs" % i
            assert not torch.isnan(a.float()).any(), "tensor %d holds unwritten rows" % i
