"""The per-layer calls of the binding: whatever arguments they are given, the library receives the same through _alcs_call and
through ctypes, or the same exception is raised.  (No GPU: the library's functions are replaced by ones that record.)"""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2109_00170_b200 import binding as B

VP, I, U = C.c_void_p, C.c_int, C.c_uint
# entry point, argument types; how the binding is called with (memory..., integers..., flags, stream)
TYPES = {"alcs_spconv1x1": [VP, VP, VP, I, I, I, VP, U, VP], "alcs_spconv1x1_ex": [VP, VP, VP, I, I, I, I, VP, VP, U, VP, VP],
         "alcs_spconv2d": [VP, VP, VP] + [I] * 8 + [VP, U, VP], "alcs_stack_run": [VP, VP]}


class Index:
    def __init__(self, v):
        self.v = v

    def __index__(self):
        return self.v


class Memory:
    def __init__(self, v):
        self.v = v

    def data_ptr(self):
        if isinstance(self.v, Exception):
            raise self.v
        return self.v


class Stream:
    def __init__(self, v):
        self.cuda_stream = v


class HasCtypes:
    ctypes = np.zeros(1).ctypes


INTEGERS = [4, np.int64(4), np.int32(-3), np.uint8(7), C.c_int(5), C.c_uint(6), Index(9), True, -1, 2 ** 31, 2 ** 40 + 3, -2 ** 63, 2 ** 64 + 1, 4.0, "4", None,
            np.float32(4), torch.tensor(3)]
MEMORY = [0, 4096, None, Memory(8192), Memory(0), Memory(np.int64(64)), Memory(None), Memory(-8), Memory(2 ** 65), Memory(ValueError("gone")),
          Memory(AttributeError("gone")), np.zeros(3), torch.zeros(3), -16, 2 ** 64 + 16, np.uint64(32), VP(48), HasCtypes(), 1.5, "x", True, np.zeros(3).ctypes]
STREAMS = [None, 0, 77, Stream(0), Stream(None), Stream(88), Stream(np.int64(3)), Stream(2 ** 64 + 1), np.int64(5), 1.0, "x", object(), True]


class Freed:
    @property
    def handle(self):
        raise B.AlcsError(B.ALCS_ERR_STATE, "freed")


class Handle:
    def __init__(self, handle):
        self.handle = handle


OBJECTS = [Handle(VP(16)), Handle(VP(None)), Handle(32), Handle(None), Freed(), object(), None]


class Library:
    """The four functions with ctypes' conversions, recording what they receive; status 0."""

    def __init__(self, calls):
        self.keep = []
        for name, types in TYPES.items():
            def record(*args, name=name):
                calls.append((name, args))
                return 0
            call = C.CFUNCTYPE(I, *types)(record)
            self.keep.append(call)
            f = C.CFUNCTYPE(I, *types)(C.cast(call, VP).value)
            f.argtypes, f.restype = types, I
            setattr(self, name, f)


def outcome(calls, f, args):
    calls.clear()
    try:
        return f(*args), list(calls)
    except Exception as e:
        return type(e), str(e), list(calls)


def variants(args, places):
    for at, values in places:
        for v in values:
            yield args[:at] + [v] + args[at + 1:]


CASES = {  # call, ordinary arguments, (place, values)...
    "spconv1x1": (B.alcs_spconv1x1, [Handle(VP(16)), 4096, 8192, 1, 2, 3, None, 1, None],
                  [(0, OBJECTS), (1, MEMORY), (2, MEMORY), (3, INTEGERS), (4, INTEGERS), (5, INTEGERS), (6, MEMORY), (7, INTEGERS), (8, STREAMS)]),
    "spconv1x1_ex": (B.alcs_spconv1x1_ex, [Handle(VP(16)), 4096, 8192, 1, 2, 3, 2, None, 64, 1, None],
                     [(0, OBJECTS), (1, MEMORY), (3, INTEGERS), (6, INTEGERS), (7, MEMORY), (8, MEMORY), (9, INTEGERS), (10, STREAMS)]),
    "spconv2d": (B.alcs_spconv2d, [Handle(VP(16)), 4096, 8192, 1, 2, 3, 4, 5, 6, 7, 8, None, 1, None],
                 [(0, OBJECTS), (2, MEMORY), (3, INTEGERS), (4, INTEGERS), (9, INTEGERS), (10, INTEGERS), (11, MEMORY), (12, INTEGERS), (13, STREAMS)]),
    "stack_run": (B.alcs_stack_run, [Handle(VP(16)), None], [(0, OBJECTS), (1, STREAMS)]),
}


@pytest.mark.parametrize("name", CASES)
def test_same_through_both_ways(monkeypatch, name):
    native = pytest.importorskip("paper_2109_00170_b200._alcs_call")
    call, ordinary, places = CASES[name]
    B.lib()                     # (binds the real functions first: the recording ones are taken back below)
    real, calls = B._lib, []
    fake = Library(calls)
    names = ("alcs_spconv1x1", "alcs_spconv1x1_ex", "alcs_spconv2d", "alcs_stack_run")
    monkeypatch.setattr(B, "_lib", fake)
    native.bind(*(C.cast(getattr(fake, n), VP).value for n in names))
    try:
        seen = 0
        for args in variants(ordinary, [(0, [ordinary[0]])] + places):
            monkeypatch.setattr(B, "_call", native)
            got = outcome(calls, call, args)
            monkeypatch.setattr(B, "_call", B._NoCall)
            assert got == outcome(calls, call, args), args
            seen += got[0] is None
        assert seen > len(places)
        # the plain form does not go through ctypes
        plain = [Handle(VP(16))] + [torch.zeros(1) if a in (4096, 8192, 64) else a for a in ordinary[1:]]
        assert getattr(native, name)(plain[0].handle, *plain[1:]) == 0 and len(calls) > 0
        assert getattr(native, name)(plain[0].handle, *plain[1:-1], np.int64(1)) is None
    finally:
        native.bind(*(C.cast(getattr(real, n), VP).value for n in names))


def test_works_without_the_helper(monkeypatch, tmp_path):
    """No _alcs_call for this Python: the library loads and every call goes through ctypes; nor does a missing compiler stop the build."""
    import sys
    import sysconfig

    import paper_2109_00170_b200 as A
    from paper_2109_00170_b200 import build
    monkeypatch.setattr(B, "_lib", None)
    monkeypatch.setattr(B, "_call", None)
    monkeypatch.delattr(A, "_alcs_call", raising=False)
    monkeypatch.setitem(sys.modules, "paper_2109_00170_b200._alcs_call", None)        # importing it raises ImportError
    assert B.lib() is not None and B._call is B._NoCall
    p = A.alcs_pack(np.ones((4, 4), np.float32), np.ones((1, 4), np.uint8), 4)
    with pytest.raises(B.AlcsError):         # (not on a device)
        A.alcs_spconv1x1(p, 4096, 8192, 1, 1, 1)
    assert build.CALL.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    monkeypatch.setattr(build, "CALL", str(tmp_path / "helper.so"))
    monkeypatch.setenv("CC", str(tmp_path / "no-such-compiler"))
    build._build_call(True)
    monkeypatch.setenv("CC", "false")
    build._build_call(True)
    assert not list(tmp_path.iterdir())
