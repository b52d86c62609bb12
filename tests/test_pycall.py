"""Argument marshalling of the binding's C extension: every kind of argument reaches the called
function as the value ctypes would have passed, errors of a conversion and of the call are raised."""
import ctypes

import pytest

from paper_2602_15318_b200 import binding as B
from paper_2602_15318_b200 import build

build.build_pycall()
from paper_2602_15318_b200 import _pycall  # noqa: E402


class _Tensor:
    def __init__(self, p):
        self.p = p

    def data_ptr(self):
        return self.p


class _Ctx:
    address = 0x7FFF12345678


class _Stream:
    cuda_stream = 77


_keep = []


def _bound(sig, status=0, lists=()):
    """A callable with signature `sig` and the list its calls are recorded in (int lists are read back)."""
    seen = []

    def record(*a):
        got = list(a)
        for k, n in lists:
            got[k] = list((ctypes.c_int32 * n).from_address(got[k])) if got[k] else None
        seen.append(got)
        return status
    cb = ctypes.CFUNCTYPE(ctypes.c_int, *[ctypes.c_int64] * len(sig))(record)
    _keep.append(cb)
    return _pycall.bind(ctypes.cast(cb, ctypes.c_void_p).value, sig, "f", B._chk), seen


@pytest.mark.parametrize("n", [0, 1, 64, 256, 257, 3000])
def test_every_kind_of_argument(n):
    _pycall.set_stream_functions(lambda: 3, lambda dev: 1000 + dev)
    fn, seen = _bound("cttiilLs", lists=[(5, n), (6, 2)])
    ints = list(range(-2, n - 2))
    fn(_Ctx(), _Tensor(2 ** 47 - 16), None, -5, 2 ** 31 - 1, ints, None, None)
    fn(_Ctx(), _Tensor(16), _Tensor(32), 1, 2, tuple(ints), (8, 9), _Stream())
    fn(_Ctx(), _Tensor(16), _Tensor(32), 1, 2, ints, [8, 9], 5)
    assert seen[0] == [_Ctx.address, 2 ** 47 - 16, 0, -5, 2 ** 31 - 1, ints, None, 1003]
    assert seen[1] == [_Ctx.address, 16, 32, 1, 2, ints, [8, 9], 77]
    assert seen[2][-1] == 5
    B._calls.__dict__.clear()                               # the binding sets its own stream functions again


def test_errors_are_raised_and_nothing_is_called():
    fn, seen = _bound("ctls")
    for bad in ((_Ctx(), _Tensor(1), None, 0), (_Ctx(), 3, [1], 0), (object(), None, [1], 0), (_Ctx(), None, ["x"], 0),
                (_Ctx(), None, [1]), (_Ctx(), None, [1], "s")):
        with pytest.raises((TypeError, AttributeError, ValueError)):
            fn(*bad)
    assert seen == []
    failing, seen = _bound("i", status=2)
    with pytest.raises(B.SparrowError) as e:
        failing(4)
    assert e.value.status == 2 and seen == [[4]]
    with pytest.raises(ValueError):
        _pycall.bind(1, "q", "f", B._chk)


def test_signatures_match_the_library():
    """One letter per argument of the C function, an int32 exactly where its ctypes prototype has one."""
    L = B.lib()
    for name, sig in B._SIGNATURES.items():
        want = getattr(L, name).argtypes
        assert len(want) == len(sig), name
        assert all((w is ctypes.c_int32) == (s == "i") for w, s in zip(want, sig)), name


@pytest.mark.parametrize("handle,want", [(0, 0), (None, 0), (5, 5), (2 ** 47 - 16, 2 ** 47 - 16)])
def test_a_stream_handle_in_a_void_pointer(handle, want):
    """What ctypes takes for a pointer argument is taken here too."""
    fn, seen = _bound("s")
    fn(ctypes.c_void_p(handle))
    assert seen == [[want]]
    for wrong in (ctypes.c_int(5), 1.5, "5"):
        with pytest.raises((TypeError, AttributeError)):
            fn(wrong)
    assert seen == [[want]]


def test_the_extension_is_built_again_for_another_torch_or_python(monkeypatch, tmp_path):
    assert build.pycall_is_current()
    monkeypatch.setattr(build, "pycall_versions", lambda: "cpython-399 torch 9.9")
    assert not build.pycall_is_current()
    monkeypatch.undo()
    monkeypatch.setattr(build, "PYCALL_VERSIONS", str(tmp_path / "none"))
    assert not build.pycall_is_current()
