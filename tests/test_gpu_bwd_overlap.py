"""The dk/dv blocks of the backward run beside its dq blocks: calls in a row equal calls with a wait behind each, bit for bit.

Few blocks (both kinds side by side), one kind short of the chip, both longer than it; every call has inputs and an angle base of its own (so
the rotation tables are written anew) but shares workspace, statistics buffers and tables with the call before, and its gradients are
read by the next kernel in the stream."""
import pytest
import torch

from paper_2509_22622_b200 import binding as B

pytestmark = pytest.mark.gpu


# heads, head_dim, tokens per frame, chunks of the clip, window in chunks
@pytest.mark.parametrize("heads,dim,p,chunks,window", [(1, 128, 1, 1, 1), (3, 128, 129, 3, 2), (2, 64, 560, 7, 6), (12, 64, 200, 4, 4),
                                                       (24, 64, 300, 3, 2), (40, 128, 496, 2, 2)])
def test_calls_in_a_row(heads, dim, p, chunks, window):
    gen = torch.Generator(device="cuda").manual_seed(p)

    def normal():
        return torch.randn(chunks * p, heads, dim, device="cuda", generator=gen).to(torch.bfloat16)

    cache = B.Cache(1, heads, dim, p, 1, 0, window + chunks - 1)
    q, k, v, q_out, out = normal(), normal(), normal(), normal(), normal()
    lse = torch.empty(heads, chunks * p, device="cuda")
    cache.clip_append_attn(0, q, k, v, 0, chunks, window, 1, p, 10000.0, q_out, out, lse)
    d_outs = [normal() for _ in range(4)]
    raw = torch.empty(B.ll_clip_backward_workspace_bytes(cache.h, chunks) + 256, dtype=torch.uint8, device="cuda")
    workspace = raw[(-raw.data_ptr()) % 256:]
    grads = [torch.empty_like(q) for _ in range(3)]

    def run(wait):
        got = []
        for i, d_out in enumerate(d_outs):
            for g in grads:
                g.fill_(float("nan"))
            shifted = lse + 0.01 * i                 # another call's statistics at another time
            B.ll_clip_attn_backward(cache.h, 0, q_out, out, d_out, shifted, 0, chunks, window, 1, p, 10000.0 / (1 + i), *grads, workspace)
            got.append([g.clone() for g in grads])   # the next kernel in the stream
            if wait:
                torch.cuda.synchronize()
        return got

    want = run(True)
    for _ in range(3):
        for a, b in zip(run(False), want):
            assert all(torch.equal(x, y) and bool(x.isfinite().all()) for x, y in zip(a, b))
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):     # captured calls, each behind the one before
        captured = run(False)
    graph.replay()
    for a, b in zip(captured, want):
        assert all(torch.equal(x, y) for x, y in zip(a, b))
    cache.check_device()
    del graph
    cache.close()
