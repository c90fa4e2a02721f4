"""Performance cases of the sink+window attention library: what is timed, on which inputs, against which tolerance.

``listed()`` names the cases, ``draw(rng)`` gives further ones of the same ranges.  For a case,
``prepare`` makes what a caller holds in hand (activations, filled caches, weights, workspaces),
``run`` is one pass through the public entry points, ``work`` the bytes and operations the pass
cannot do without, ``tolerance`` how far another correct implementation of the same precision
may be off, and ``exact`` what the pass returns in plain 64-bit arithmetic.  Sizes are those of the benchmark workloads of ``synth.CONFIGS`` and generic ones.

Kinds of pass:
  decode    one denoising pass of a stream's newest chunk in one layer: rotate q and k (with the
            q/k norm in front when the case says so), write k and v over the chunk's rows, attend
            over the sink and the window.  All but one pass of a chunk are such overwrites.
  append    the front end of that pass alone, for callers that attend elsewhere in their graph
  project   the layer's QKV projection with the front end in its epilogue
  batched   a serving step: the newest chunks of several streams, attended in one launch
  recache   a prompt switch: every resident window frame rebuilt and attended block-causally
  clip      forward of a training clip behind its context (also the prefill of a stream)
  backward  gradients of that clip
  cross     the video tokens of a chunk over the prompt's tokens
"""
import math

import torch

from paper_2509_22622_b200 import binding as B

THETA = 10000.0
BF16 = torch.bfloat16
WAN = dict(heads=12, head_dim=128, grid_h=30, grid_w=52, chunk=3, sink=3, window=9)
# Attention flops that bound a drawn case: below the backward pass of the 21-frame clip, and lower
# for heads of 64, whose exponentials cost twice as much per flop.
MAX_FLOPS = {128: 4e12, 64: 2e12}


def listed():
    return [
        # the smallest stream of the test-suite: launches and host time are all there is
        dict(name="tiny_decode", kind="decode", heads=2, head_dim=64, grid_h=4, grid_w=4, chunk=1, sink=1, window=2,
             filled=5, norm=False, kv="bf16"),
        # a preview-sized stream, 493 tokens per frame: ragged tiles, fewer columns than the GPU has SMs
        dict(name="preview_decode", kind="decode", heads=12, head_dim=128, grid_h=17, grid_w=29, chunk=3, sink=3,
             window=9, filled=6, norm=False, kv="bf16"),
        # the benchmark layer (832x480 video, 4680 queries over 18720 keys) in its steady state
        dict(WAN, name="layer_decode", kind="decode", filled=6, norm=False, kv="bf16"),
        # the same over the 8-bit cache
        dict(WAN, name="layer_decode_8bit", kind="decode", filled=6, norm=False, kv="e4m3"),
        # the same width in 24 heads of 64
        dict(WAN, name="layer_decode_head64", kind="decode", heads=24, head_dim=64, filled=6, norm=False, kv="bf16"),
        # the front end with the q/k norm, for a caller with its own projection
        dict(WAN, name="layer_append_norm", kind="append", filled=6, norm=True, kv="bf16"),
        # the projection of the layer (model width 1536) with norm, rotation and append
        dict(WAN, name="layer_project_norm", kind="project", filled=6, norm=True, d_model=1536),
        # serving: eight streams from their first chunk to their 51st, activations with outliers
        dict(WAN, name="serve_8_streams", kind="batched", positions="0,1,2,3,6,13,29,50", outliers=0.01),
        # prompt switch with a full window
        dict(WAN, name="layer_recache", kind="recache", filled=6),
        # training clip of 21 frames behind a full window: forward, then backward
        dict(WAN, name="clip_forward", kind="clip", window=27, filled=4, clip_chunks=7, attn_window=9),
        dict(WAN, name="clip_backward", kind="backward", window=27, filled=4, clip_chunks=7, attn_window=9),
        # cross-attention of a chunk to a padded 512-token prompt
        dict(name="prompt_cross", kind="cross", heads=12, head_dim=128, n_q=4680, n_k=512),
    ]


def _log(rng, lo, hi):
    """A whole number of [lo, hi], evenly over the logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: any kind, 1 to 40 heads, grids from 4x4 to 45x80, chunks of 1 to 4 frames, windows of 1 to 6
    chunks, streams from their first chunk on, every cache format and front end."""
    while True:
        kind = rng.choice(("decode", "decode", "append", "project", "batched", "recache", "clip", "backward", "cross"))
        c = dict(kind=kind, heads=rng.choice((1, 2, 3, 6, 8, 12, 16, 24, 40)), head_dim=rng.choice((64, 128, 128)))
        if kind == "cross":
            c.update(n_q=_log(rng, 16, 16384), n_k=_log(rng, 16, 4096))
        else:
            chunk = rng.randint(1, 4)
            c.update(grid_h=_log(rng, 4, 45), grid_w=_log(rng, 4, 80), chunk=chunk, sink=chunk * rng.randint(0, 2),
                     window=chunk * rng.randint(1, 6))
        if kind in ("decode", "append", "project", "recache"):
            c["filled"] = rng.randint(1, 12)
        if kind in ("decode", "append"):
            c["norm"] = rng.random() < 0.5
            c["kv"] = "bf16" if c["norm"] else rng.choice(("bf16", "e4m3"))
        if kind == "project":
            c["norm"] = rng.random() < 0.7
            c["d_model"] = 8 * _log(rng, 16, 640)
            width = c["heads"] * c["head_dim"]
            if width % 256 and width % 192:
                continue
        if kind == "batched":
            c["positions"] = ",".join(str(_log(rng, 1, 60) - 1) for _ in range(rng.randint(2, 8)))
            c["outliers"] = rng.choice((0.0, 0.01))
        if kind in ("clip", "backward"):
            c["clip_chunks"] = rng.randint(2, 7)
            c["attn_window"] = c["window"]
            c["window"] += (c["clip_chunks"] - 1) * c["chunk"]
            c["filled"] = rng.randint(0, 6)
        if kind == "recache" and _recached_frames(c) == 0:
            continue
        w = work(c)
        if w["flops"] <= MAX_FLOPS[c["head_dim"]] and w["bytes"] <= 1e9 and _tokens(c) * c["heads"] * c["head_dim"] <= 1 << 27:
            return c


# ---- shapes -------------------------------------------------------------------------------

def _tokens(c):
    """Query tokens of a pass."""
    if c["kind"] == "cross":
        return c["n_q"]
    p = c["chunk"] * c["grid_h"] * c["grid_w"]
    if c["kind"] == "batched":
        return p * len(_positions(c))
    if c["kind"] in ("clip", "backward"):
        return p * c["clip_chunks"]
    if c["kind"] == "recache":
        return _recached_frames(c) * c["grid_h"] * c["grid_w"]
    return p


def _positions(c):
    return [int(x) for x in c["positions"].split(",")]


def _recached_frames(c):
    end = c["filled"] * c["chunk"]
    return end - max(c["sink"], end - c["window"]) if end > c["sink"] else 0


def _seen(c, end, window, first=0, since=0):
    """Frames a chunk that ends in front of frame `end` sees: the sink and of the window those from `first` on.
    Only frames from `since` on are counted."""
    lo = max(c["sink"], end - window, first, since)
    return max(0, min(c["sink"], end) - since) + max(0, end - lo)


def _attention_groups(c):
    """(queries, keys) of every chunk of queries of the pass."""
    kind = c["kind"]
    if kind in ("append", "project"):
        return []
    if kind == "cross":
        return [(c["n_q"], c["n_k"])]
    p, n = c["grid_h"] * c["grid_w"], c["chunk"]
    if kind == "decode":
        ends, window, first = [c["filled"] * n], c["window"], 0
    elif kind == "batched":
        ends, window, first = [(x + 1) * n for x in _positions(c)], c["window"], 0
    elif kind == "recache":
        end, frames = c["filled"] * n, _recached_frames(c)
        ends, window, first = [end - frames + (g + 1) * n for g in range(frames // n)], c["window"], end - frames
    else:
        ends, window, first = [(c["filled"] + g + 1) * n for g in range(c["clip_chunks"])], c["attn_window"], 0
    return [(n * p, _seen(c, e, window, first) * p) for e in ends]


def work(case):
    """Bytes and floating-point operations a pass cannot do without."""
    kind, width = case["kind"], case["heads"] * case["head_dim"]
    row = 2 * width                                          # one token of q, k or v, or of an output, in bf16
    tokens, groups = _tokens(case), _attention_groups(case)
    flops = sum(4.0 * nq * nk * width for nq, nk in groups)
    if kind == "cross":
        return {"bytes": float(row * (2 * tokens + 2 * case["n_k"])), "flops": flops}
    p = case["grid_h"] * case["grid_w"]
    stored = width * (1 if case.get("kv") == "e4m3" else 2)  # one token of K or V as the cache holds it
    if kind == "project":
        d = case["d_model"]
        return {"bytes": float(2 * d * (tokens + 3 * width) + row * tokens + 2 * stored * tokens),
                "flops": 2.0 * tokens * d * 3 * width}
    front = tokens * (4 * row + 2 * stored)                  # q, k, v in; rotated q and the cache rows out
    if kind == "append":
        return {"bytes": float(front), "flops": 12.0 * tokens * width}
    if kind == "backward":
        # S, dP and dq run over all visible keys, dk and dv over the clip's own
        n, start = case["chunk"], case["filled"] * case["chunk"]
        own = sum(nq * _seen(case, start + (g + 1) * n, case["attn_window"], since=start) * p for g, (nq, _) in enumerate(groups))
        flops = 2.0 * width * (3 * sum(nq * nk for nq, nk in groups) + 2 * own)
        seen = tokens + min(case["filled"] * case["chunk"], case["sink"] + case["attn_window"]) * p
        return {"bytes": float(row * (3 * tokens + 3 * tokens + 2 * seen) + 4 * tokens * case["heads"]), "flops": flops}
    if kind == "batched":
        old = sum(nk - nq for nq, nk in groups)
    elif kind == "clip":
        old = min(case["filled"] * case["chunk"], case["sink"] + case["attn_window"]) * p
    else:
        old = max(nk for _, nk in groups) - tokens
    return {"bytes": float(front + row * tokens + 2 * stored * max(0, old)), "flops": flops}


def tolerance(case):
    """About four times what one implementation is off from the same call in 64-bit arithmetic on the stored operands."""
    if case["kind"] in ("append", "project"):
        t = {"rel": 7e-3, "max": 1.6e-2}                     # one rounding to bf16: measured rel 1.7e-3, max 3.9e-3
    else:
        t = {"rel": 1e-2, "max": 7e-2}                       # weights and results in bf16: measured rel 2.4e-3, max 1.7e-2
    if case.get("kv") == "e4m3":
        t["differ"] = 1e-3                                   # a code on a rounding boundary may fall either way
    return t


# ---- inputs and passes ----------------------------------------------------------------------

class _Inputs:
    """Seeded activations on the GPU: normal, as behind a q/k norm, with rare large entries where asked."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)

    def normal(self, *shape, outliers=0.0, scale=1.0):
        x = torch.randn(*shape, device="cuda", generator=self.gen)
        if outliers:
            x = torch.where(torch.rand(*shape, device="cuda", generator=self.gen) < outliers, 20.0 * x, x)
        return (x * scale).to(BF16)

    def floats(self, *shape, mean=0.0, std=1.0):
        return mean + std * torch.randn(*shape, device="cuda", generator=self.gen)


def _cache(c, window=None):
    cache = B.Cache(1, c["heads"], c["head_dim"], c["grid_h"] * c["grid_w"], c["chunk"], c["sink"],
                    window or c["window"], kv_format=B.LL_KV_E4M3 if c.get("kv") == "e4m3" else B.LL_KV_BF16)
    if c.get("kv") == "e4m3":
        cache.set_kv_scales(0, [6.0 / 448.0] * c["heads"], [6.0 / 448.0] * c["heads"])
    return cache


def _fill(cache, c, inputs, chunks, outliers=0.0):
    """Append `chunks` chunks.  Only what is still resident at the end needs contents of its own."""
    shape = (c["chunk"] * c["grid_h"] * c["grid_w"], c["heads"], c["head_dim"])
    kv = None
    for i in range(chunks):
        if kv is None or i * c["chunk"] < c["sink"] or (chunks - i) * c["chunk"] <= cache.W:
            kv = inputs.normal(*shape, outliers=outliers), inputs.normal(*shape, outliers=outliers)
        cache.rope_append_kv(0, None, kv[0], kv[1], i * c["chunk"], c["grid_h"], c["grid_w"], THETA)


def _stored(cache):
    return {"k": cache.kv_view(0, 0), "v": cache.kv_view(0, 1)}


def _workspace(nbytes):
    raw = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    return raw[(-raw.data_ptr()) % 256:]


def prepare(case, seed):
    c, kind = case, case["kind"]
    inputs = _Inputs(seed)
    s = {"case": c}
    if kind == "cross":
        # the handle only lends its scratch
        s["cache"] = B.Cache(1, c["heads"], c["head_dim"], 16, 1, 1, 1)
        s["q"] = inputs.normal(c["n_q"], c["heads"], c["head_dim"])
        s["k"], s["v"] = (inputs.normal(c["n_k"], c["heads"], c["head_dim"]) for _ in range(2))
        s["out"] = torch.empty_like(s["q"])
        return s
    p, n, width = c["grid_h"] * c["grid_w"], c["chunk"], c["heads"] * c["head_dim"]

    def activations(frames, outliers=0.0):
        return tuple(inputs.normal(frames * p, c["heads"], c["head_dim"], outliers=outliers) for _ in range(3))

    if kind == "batched":
        s["streams"] = []
        for pos in _positions(c):
            cache = _cache(c)
            _fill(cache, c, inputs, pos + 1, c["outliers"])
            q, k, v = activations(n, c["outliers"])
            s["streams"].append(dict(cache=cache, start=pos * n, q=q, k=k, v=v, q_out=torch.empty_like(q),
                                     out=torch.empty_like(q), stored=_stored(cache)))
        s["items"] = [(t["cache"], 0, t["q_out"], t["start"], t["out"], None) for t in s["streams"]]
        return s

    cache = s["cache"] = _cache(c)
    _fill(cache, c, inputs, c["filled"])
    s["start"] = (c["filled"] - 1) * n
    s["stored"] = _stored(cache)
    if kind == "project":
        s["x"] = inputs.normal(n * p, c["d_model"])
        s["w"] = inputs.normal(3 * width, c["d_model"], scale=c["d_model"] ** -0.5)
        s["bias"] = inputs.floats(3 * width, std=0.1)
        s["q_out"] = torch.empty(n * p, c["heads"], c["head_dim"], device="cuda", dtype=BF16)
        s["gain_q"] = s["gain_k"] = s["row_scale"] = s["ws"] = None
        if c["norm"]:
            s["gain_q"], s["gain_k"] = (inputs.floats(width, mean=1.0, std=0.1) for _ in range(2))
            s["row_scale"] = torch.empty(n * p, device="cuda")
            s["ws"] = _workspace(B.ll_qkv_proj_workspace_bytes(cache.h))
        return s
    if kind in ("decode", "append"):
        s["q"], s["k"], s["v"] = activations(n)
        if c["norm"]:
            s["gain_q"], s["gain_k"] = (inputs.floats(width, mean=1.0, std=0.1) for _ in range(2))
    elif kind == "recache":
        s["frames"] = _recached_frames(c)
        s["q"], s["k"], s["v"] = activations(s["frames"])
    else:
        s["frames"] = c["clip_chunks"] * n
        s["start"] = c["filled"] * n
        s["q"], s["k"], s["v"] = activations(s["frames"])
        s["lse"] = torch.empty(c["heads"], s["frames"] * p, device="cuda")
    s["q_out"], s["out"] = torch.empty_like(s["q"]), torch.empty_like(s["q"])
    if kind == "backward":
        cache.clip_append_attn(0, s["q"], s["k"], s["v"], s["start"], s["frames"], c["attn_window"], c["grid_h"],
                               c["grid_w"], THETA, s["q_out"], s["out"], s["lse"])
        s["d_out"] = inputs.normal(*s["q"].shape)
        s["dq"], s["dk"], s["dv"] = (torch.empty_like(s["q"]) for _ in range(3))
        s["ws"] = _workspace(B.ll_clip_backward_workspace_bytes(cache.h, s["frames"]))
    return s


def _front(s, c, cache, start, q, k, v, q_out):
    if c.get("norm"):
        cache.norm_rope_append_kv(0, q, k, v, s["gain_q"], s["gain_k"], 1e-6, start, c["grid_h"], c["grid_w"], THETA, q_out)
    else:
        cache.rope_append_kv(0, q, k, v, start, c["grid_h"], c["grid_w"], THETA, q_out)


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "cross":
        s["cache"].cross_attn(s["q"], s["k"], s["v"], s["out"])
        return s["out"]
    if kind == "batched":
        for t in s["streams"]:
            _front(s, c, t["cache"], t["start"], t["q"], t["k"], t["v"], t["q_out"])
        B.Cache.sink_window_attn_batched(s["items"])
        return [[t["out"], t["q_out"], t["stored"]] for t in s["streams"]]
    cache = s["cache"]
    if kind == "project":
        B.ll_qkv_proj_append(cache.h, 0, s["x"], s["w"], s["bias"], s["gain_q"], s["gain_k"], 1e-6, s["start"], c["chunk"],
                             c["grid_h"], c["grid_w"], THETA, s["q_out"], s["row_scale"], s["ws"])
        return [s["q_out"], s["row_scale"], s["stored"]]
    if kind == "append":
        _front(s, c, cache, s["start"], s["q"], s["k"], s["v"], s["q_out"])
        return [s["q_out"], s["stored"]]
    if kind == "decode":
        _front(s, c, cache, s["start"], s["q"], s["k"], s["v"], s["q_out"])
        cache.sink_window_attn(0, s["q_out"], s["start"], s["out"])
        return [s["out"], s["q_out"], s["stored"]]
    if kind == "recache":
        cache.recache(0, s["q"], s["k"], s["v"], s["frames"], c["grid_h"], c["grid_w"], THETA, s["q_out"], s["out"])
        return [s["out"], s["q_out"], s["stored"]]
    if kind == "clip":
        # the stream moves on: the next clip stands behind this one
        cache.clip_append_attn(0, s["q"], s["k"], s["v"], s["start"], s["frames"], c["attn_window"], c["grid_h"],
                               c["grid_w"], THETA, s["q_out"], s["out"], s["lse"])
        s["start"] += s["frames"]
        return [s["out"], s["lse"], s["q_out"], s["stored"]]
    B.ll_clip_attn_backward(cache.h, 0, s["q_out"], s["out"], s["d_out"], s["lse"], s["start"], s["frames"], c["attn_window"],
                            c["grid_h"], c["grid_w"], THETA, s["dq"], s["dk"], s["dv"], s["ws"])
    return [s["dq"], s["dk"], s["dv"]]


# ---- the same passes in plain torch, 64 bits ---------------------------------------------------
#
# What the library stores in 16 or 8 bits on the way (rotated q and k, cache rows, the forward's
# output that the backward is handed) is rounded here as well, so that what is left is the error
# of the arithmetic and of the last rounding.

MAX_SCORES = 1 << 26                                         # score entries held at a time


def _round(x):
    return x.to(BF16).double()


def _rotation(c, start, frames):
    """(cos, sin) [tokens, 1, pairs] of the frames' tokens: the pairs of a head row go to t, then h, then w."""
    n_h = c["head_dim"] // 6
    n_t = c["head_dim"] // 2 - 2 * n_h

    def axis(n, pairs):
        i = torch.arange(pairs, device="cuda", dtype=torch.float64)
        return n.double()[:, None] * THETA ** (-i / pairs)

    at = torch.arange(frames * c["grid_h"] * c["grid_w"], device="cuda")
    p = c["grid_h"] * c["grid_w"]
    angle = torch.cat([axis(start + at // p, n_t), axis(at % p // c["grid_w"], n_h), axis(at % c["grid_w"], n_h)], 1)
    return angle.cos()[:, None], angle.sin()[:, None]


def _rotate(x, cos, sin):
    a, b = x[..., 0::2], x[..., 1::2]
    return torch.stack([a * cos - b * sin, a * sin + b * cos], -1).flatten(-2)


class _PlainCache:
    """Sink and ring of one layer, [row, head, dim]."""

    def __init__(self, c):
        self.c, self.W = c, c["window"]
        self.p = c["grid_h"] * c["grid_w"]
        shape = ((c["sink"] + self.W) * self.p, c["heads"], c["head_dim"])
        self.k, self.v = (torch.zeros(*shape, device="cuda", dtype=torch.float64) for _ in range(2))

    def rows(self, frames):
        s = self.c["sink"]
        first = torch.tensor([f if f < s else s + (f - s) % self.W for f in frames], device="cuda")
        return (first[:, None] * self.p + torch.arange(self.p, device="cuda")).flatten()

    def _stored(self, x):
        if self.c.get("kv") != "e4m3":
            return _round(x)
        scale = torch.tensor(6.0 / 448.0, dtype=torch.float32, device="cuda").double()
        return (x / scale).clamp(-448, 448).float().to(torch.float8_e4m3fn).double() * scale

    def put(self, k, v, start):
        """Rows that are rotated already."""
        at = self.rows(range(start, start + len(k) // self.p))
        self.k[at], self.v[at] = self._stored(k), self._stored(v)

    def rope_append_kv(self, layer, q, k, v, start, grid_h, grid_w, theta):
        self.put(_rotate(k.double(), *_rotation(self.c, start, self.c["chunk"])), v.double(), start)

    def visible(self, end, window, first=0):
        return self.rows(list(range(min(self.c["sink"], end))) + list(range(max(self.c["sink"], end - window, first), end)))

    def stored(self):
        if self.c.get("kv") == "e4m3":
            return {"k": None, "v": None}                    # codes: whole values
        return {"k": self.k.transpose(0, 1), "v": self.v.transpose(0, 1)}


def _attend(q, k, v):
    """softmax(q k^T / sqrt(D)) v and the log of the sums, [rows, heads, D] and [heads, rows]."""
    out, lse = torch.empty_like(q), torch.empty(q.shape[1], q.shape[0], device="cuda", dtype=torch.float64)
    step = max(1, MAX_SCORES // len(k))
    for h in range(q.shape[1]):
        for i in range(0, len(q), step):
            s = q[i:i + step, h] @ k[:, h].T * q.shape[2] ** -0.5
            lse[h, i:i + step] = s.logsumexp(1)
            out[i:i + step, h] = (s - lse[h, i:i + step, None]).exp_() @ v[:, h]
    return out, lse


def _attend_groups(cache, q, starts, window, first=0):
    n = cache.c["chunk"] * cache.p
    parts = []
    for g, start in enumerate(starts):
        at = cache.visible(start + cache.c["chunk"], window, first)
        parts.append(_attend(q[g * n:(g + 1) * n], cache.k[at], cache.v[at]))
    return torch.cat([o for o, _ in parts]), torch.cat([x for _, x in parts], 1)


def _gradients(cache, q, out, d_out, lse, starts, window):
    c, n = cache.c, cache.c["chunk"] * cache.p
    dq, dk, dv = torch.zeros_like(q), torch.zeros_like(cache.k), torch.zeros_like(cache.v)
    delta, scale = (out * d_out).sum(2), c["head_dim"] ** -0.5
    for g, start in enumerate(starts):
        at = cache.visible(start + c["chunk"], window)
        step = max(1, MAX_SCORES // len(at))
        for h in range(c["heads"]):
            k, v = cache.k[at, h], cache.v[at, h]
            dk_h, dv_h = torch.zeros_like(k), torch.zeros_like(v)
            for i in range(g * n, (g + 1) * n, step):
                rows = slice(i, min(i + step, (g + 1) * n))
                w = (q[rows, h] @ k.T * scale - lse[h, rows, None]).exp_()
                ds = w * (d_out[rows, h] @ v.T - delta[rows, h, None])
                dq[rows, h] = ds @ k * scale
                dk_h += ds.T @ q[rows, h] * scale
                dv_h += w.T @ d_out[rows, h]
            dk[at, h] += dk_h
            dv[at, h] += dv_h
    own = cache.rows(range(starts[0], starts[-1] + c["chunk"]))
    cos, sin = _rotation(c, starts[0], len(starts) * c["chunk"])
    return [_rotate(dq, cos, -sin), _rotate(dk[own], cos, -sin), dv[own]]


def _rms(x, eps=1e-6):
    return (x.flatten(1).square().mean(1) + eps).rsqrt()


def exact(case, seed):
    """What `run` returns on `prepare(case, seed)`: draws the inputs in the same order."""
    c, kind = case, case["kind"]
    inputs = _Inputs(seed)
    if kind == "cross":
        q = inputs.normal(c["n_q"], c["heads"], c["head_dim"])
        k, v = (inputs.normal(c["n_k"], c["heads"], c["head_dim"]) for _ in range(2))
        return _attend(q.double(), k.double(), v.double())[0]
    p, n, heads, dim = c["grid_h"] * c["grid_w"], c["chunk"], c["heads"], c["head_dim"]

    def activations(frames, outliers=0.0):
        return tuple(inputs.normal(frames * p, heads, dim, outliers=outliers).double() for _ in range(3))

    if kind == "batched":
        outs = []
        for pos in _positions(c):
            cache = _PlainCache(c)
            _fill(cache, c, inputs, pos + 1, c["outliers"])
            q, k, v = activations(n, c["outliers"])
            turn = _rotation(c, pos * n, n)
            cache.put(_rotate(k, *turn), v, pos * n)
            q = _rotate(q, *turn)
            outs.append([_attend_groups(cache, _round(q), [pos * n], c["window"])[0], q, cache.stored()])
        return outs

    cache = _PlainCache(c)
    _fill(cache, c, inputs, c["filled"])
    start = (c["filled"] - 1) * n
    if kind == "project":
        width = heads * dim
        x = inputs.normal(n * p, c["d_model"]).double()
        w = inputs.normal(3 * width, c["d_model"], scale=c["d_model"] ** -0.5).double()
        y = x @ w.T + inputs.floats(3 * width, std=0.1).double()
        q, k, v = (t.reshape(n * p, heads, dim) for t in y.chunk(3, 1))
        row_scale = None
        if c["norm"]:
            gain_q, gain_k = (inputs.floats(width, mean=1.0, std=0.1).double().reshape(heads, dim) for _ in range(2))
            row_scale, k_scale = _rms(q), _rms(k)
            q, k = q * gain_q, k * gain_k * k_scale[:, None, None]
        turn = _rotation(c, start, n)
        cache.put(_rotate(k, *turn), v, start)
        return [_rotate(q, *turn), row_scale, cache.stored()]
    frames = n
    if kind == "recache":
        frames = _recached_frames(c)
        start = c["filled"] * n - frames
    elif kind in ("clip", "backward"):
        frames, start = c["clip_chunks"] * n, c["filled"] * n
    q, k, v = activations(frames)
    if c.get("norm"):
        gain_q, gain_k = (inputs.floats(heads * dim, mean=1.0, std=0.1).double().reshape(heads, dim) for _ in range(2))
        q, k = q * gain_q * _rms(q)[:, None, None], k * gain_k * _rms(k)[:, None, None]
    turn = _rotation(c, start, frames)
    cache.put(_rotate(k, *turn), v, start)
    q = _rotate(q, *turn)
    if kind == "append":
        return [q, cache.stored()]
    starts = range(start, start + frames, n)
    window, first = c.get("attn_window", c["window"]), start if kind == "recache" else 0
    out, lse = _attend_groups(cache, _round(q), starts, window, first)
    if kind == "clip":
        return [out, lse, q, cache.stored()]
    if kind == "backward":
        return _gradients(cache, _round(q), _round(out), inputs.normal(frames * p, heads, dim).double(), lse, starts, window)
    return [out, q, cache.stored()]
