"""CPU-only: the marshalling module takes, refuses and answers what the ctypes functions do."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2509_22622_b200 import binding as B


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2509_22622_b200 import build
    build.build()
    B.lib()
    assert B._fast is not None, "the marshalling module has not been built"


@pytest.fixture(params=["module", "ctypes"])
def way(request, monkeypatch):
    if request.param == "ctypes":
        monkeypatch.setattr(B, "_fast", None)
    return request.param


X = torch.zeros(32, 2, 64, dtype=torch.bfloat16)
GAIN = torch.ones(128)


def handle():
    h = B.ll_cache_create(1, 2, 64, 16, 2, 2, 4)
    B.ll_cache_set_dry_run(h, True)
    return h


def outcome(call):
    try:
        return call()
    except B.LLError as e:
        return e.code, str(e)
    except Exception:                                  # of the marshalling, whatever its type
        return "refused"


# name, arguments behind the handle
CALLS = {
    "ll_rope_append_kv": (0, X, X, X, 0, 2, 4, 4, 10000.0, X, 0),
    "ll_norm_rope_append_kv": (0, X, X, X, GAIN, GAIN, 1e-6, 0, 2, 4, 4, 10000.0, X, 0),
    "ll_sink_window_attn": (0, X, 0, 2, X, None, 0),
    "ll_cross_attn": (X, X, X, X, None, 0),
    "ll_qkv_proj_append": (0, X.reshape(32, 128), X, None, GAIN, GAIN, 1e-6, 0, 2, 4, 4, 10000.0, X, GAIN, GAIN, 0),
}


def answers(way_is):
    """What every call answers with one argument at a time replaced."""
    got = []
    for name, args in CALLS.items():
        fn = getattr(B, name)
        for i in range(-2, len(args)):
            for other in (None, -1, 7, 1 << 33, 2.5, True, "x", X, np.int64(1), np.float32(3.0)):
                h = handle()
                if name == "ll_sink_window_attn":
                    B.ll_rope_append_kv(h, *CALLS["ll_rope_append_kv"])
                a = list(args)
                if i >= 0:
                    a[i] = other
                use = h if i != -2 else None if other is None else ctypes.c_void_p(None)
                if i == -1:
                    use = h.value
                got.append((name, i, repr(other)[:20], outcome(lambda: fn(use, *a)), B.ll_cache_get_state(h).end))
                B.ll_cache_destroy(h)
    return got


def test_same_answers(monkeypatch):
    native = answers("module")
    monkeypatch.setattr(B, "_fast", None)
    plain = answers("ctypes")
    assert native == plain
    assert {type(x[3]) for x in native} == {type(None), tuple, str}           # taken, refused by the library, refused on the way


class Value:
    def __init__(self, value):
        self.value = value


class Handle(ctypes.c_void_p):
    pass


def test_same_handles(way):
    """A handle is an integer or a c_void_p; other things with an address in them are refused before the library sees it."""
    for name, args in CALLS.items():
        fn = getattr(B, name)
        for kind in (ctypes.c_long, ctypes.c_ulong, ctypes.c_uint64, Value):
            h = handle()
            with pytest.raises(ctypes.ArgumentError):
                fn(kind(h.value), *args)
            with pytest.raises((TypeError, ctypes.ArgumentError)):
                B.ll_sink_window_attn_batched([(kind(h.value), 0, X, 0, 2, X, None)], 0)
            B.ll_cache_destroy(h)
        for kind in (int, ctypes.c_void_p, Handle):
            h = handle()
            assert outcome(lambda: fn(kind(h.value), *args)) != "refused"
            B.ll_cache_destroy(h)


def test_batched(way):
    hs = [handle() for _ in range(9)]
    for h in hs:
        B.ll_rope_append_kv(h, *CALLS["ll_rope_append_kv"])
    item = lambda h: (h, 0, X, 0, 2, X, None)
    assert B.ll_sink_window_attn_batched([item(h) for h in hs[:8]], 0) is None
    assert B.ll_sink_window_attn_batched(tuple(item(h) for h in hs[:8]), 0) is None
    assert [B.ll_cache_get_state(h).n_attn_calls for h in hs] == [2] * 8 + [0]
    for bad in ([], [item(h) for h in hs], [item(hs[0]), item(hs[0])], [(None,) + item(hs[0])[1:]]):
        with pytest.raises(B.LLError):
            B.ll_sink_window_attn_batched(bad, 0)
    with pytest.raises((TypeError, ValueError, ctypes.ArgumentError)):
        B.ll_sink_window_attn_batched([item(hs[0])[:6]], 0)
    for h in hs:
        B.ll_cache_destroy(h)


@pytest.mark.parametrize("cc,built", [("gcc -m64", True), ("no-such-compiler", False), ("false", False), ("gcc '", False)])
def test_the_compiler_of_the_environment(cc, built, monkeypatch, tmp_path, capfd):
    """CC may come with options; one that does not do leaves the module out, an older one too, and does not end the build."""
    from paper_2509_22622_b200 import build
    module = tmp_path / "_marshal.so"
    module.write_bytes(b"older")
    monkeypatch.setattr(build, "MARSHAL", str(module))
    monkeypatch.setenv("CC", cc)
    build.build_marshal(force=True)
    assert module.exists() == built and (not built or module.read_bytes() != b"older")
    assert ("has not been built" in capfd.readouterr().err) != built
    assert [f.name for f in tmp_path.iterdir()] == ["_marshal.so"] * built


def test_errors_are_reported(way):
    h = handle()
    with pytest.raises(B.LLError, match="grid"):
        B.ll_rope_append_kv(h, 0, X, X, X, 0, 2, 5, 4, 10000.0, X, 0)
    B.ll_cache_destroy(h)
