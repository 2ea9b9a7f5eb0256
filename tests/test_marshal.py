"""The C marshalling of the hot calls hands on exactly what it was given (needs no device: the entry points are
replaced by recording callbacks, the tensors by objects with data_ptr() and stride())."""

import ctypes as C

import pytest


class Fake:
    def __init__(self, ptr, stride=(4096, 1024, 128, 1)):
        self.ptr, self.st = ptr, stride

    def data_ptr(self):
        return self.ptr

    def stride(self):
        return self.st


@pytest.fixture()
def recorded():
    from paper_2503_08879_b200 import binding as B
    vp, i32, i64 = C.c_void_p, C.c_int32, C.c_int64
    sigs = {"score": (vp, vp, vp, B.Strides, i64, i32, i32, vp, i64, vp),
            "select_compact": (vp, vp, i64, vp, vp, B.Strides, i64, i32, i32, i32, vp, vp, vp, B.Strides, C.POINTER(B.CacheState), vp),
            "decode_attn": (vp, vp, vp, vp, vp, vp, B.Strides, C.POINTER(B.CacheState), vp, vp, vp),
            "pool_scores": (vp, vp, i64, i64, i32, i32, vp, i64, vp),
            "quest_bounds": (vp, vp, vp, vp, i64, vp, i64, vp),
            "select_topk": (vp, vp, i64, i64, i32, vp, vp)}
    got, keep = [], []

    def plain(x):
        if isinstance(x, B.Strides):
            return x.batch_stride, x.head_stride, x.token_stride
        if hasattr(x, "contents"):
            x.contents.len += 1                                  # the callee writes into the caller's structure
            return x.contents.k_q
        return x

    def record(*a):
        got.append(tuple(plain(x) for x in a))
        return -3

    for s in sigs.values():
        keep.append(C.CFUNCTYPE(C.c_int, *s)(record))
    B._marshal.bind(*(C.cast(f, vp).value for f in keep), lambda: 77, C.ArgumentError)
    yield B, got
    B._marshal.bind(*(C.cast(getattr(B.lib, "sagekv_" + n), vp).value for n in sigs), B._stream_handle, C.ArgumentError)


def test_every_argument_arrives(recorded):
    B, got = recorded
    m, ctx, K, V = B._marshal, C.c_void_p(9), Fake(3, (1 << 40, -8, 256, 1)), Fake(4)
    st = B.CacheState(1, 2, 3, 4, 5, 6, None)
    assert m.score(ctx, Fake(2), K, 1 << 33, -1, 7, Fake(5), 12) == -3
    assert m.select_compact(ctx, None, 8, K, V, 100, 4, 5, 6, Fake(10), Fake(11, (3, 2, 1, 1)), Fake(12), st) == -3
    assert m.decode_attn(None, Fake(2), None, None, K, V, st, Fake(6), None) == -3
    assert m.pool_scores(ctx, Fake(1), 2, 3, 4, 5, Fake(6), 7) == -3
    assert m.quest_bounds(ctx, Fake(1), Fake(2), Fake(3), 4, Fake(5), 6) == -3
    assert m.select_topk(ctx, Fake(1), 2, 3, 4, Fake(5)) == -3
    k = (1 << 40, -8, 256)
    assert got == [(9, 2, 3, k, 1 << 33, -1, 7, 5, 12, 77),
                   (9, None, 8, 3, 4, k, 100, 4, 5, 6, 10, 11, 12, (3, 2, 1), 2, 77),
                   (None, 2, None, None, 3, 4, k, 2, 6, None, 77),
                   (9, 1, 2, 3, 4, 5, 6, 7, 77),
                   (9, 1, 2, 3, 4, 5, 6, 77),
                   (9, 1, 2, 3, 4, 5, 77)]
    assert st.len == 8                                           # both calls that take it saw this very structure


def test_wrong_arguments_raise(recorded):
    B, got = recorded
    m, ctx, K = B._marshal, C.c_void_p(9), Fake(3)
    with pytest.raises(C.ArgumentError):
        m.score(ctx, Fake(2), K, 1.5, 0, 0, Fake(5), 12)
    with pytest.raises(ValueError):
        m.score(ctx, Fake(2), Fake(3, (1, 2, 3)), 1, 0, 0, Fake(5), 12)
    with pytest.raises(ValueError):
        m.score(ctx, Fake(2), Fake(3, (1, 2, 3, 2)), 1, 0, 0, Fake(5), 12)
    with pytest.raises(AttributeError):
        m.score(ctx, Fake(2), 5, 1, 0, 0, Fake(5), 12)
    with pytest.raises(TypeError):
        m.decode_attn(ctx, Fake(2), None, None, K, K, object(), Fake(6), None)
    with pytest.raises(TypeError):
        m.score(ctx)
    assert got == []


def test_the_module_belongs_to_this_interpreter():
    """Another Python version must not take the module for its own: its name carries the tag of the one it was built for."""
    import sysconfig
    from paper_2503_08879_b200 import binding as B
    assert B._marshal.__file__.endswith("_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))
