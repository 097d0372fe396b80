"""Argument conversion of the forward calls, by the extension module and by ctypes, through calls that the library refuses before it
touches a GPU, and the module's independence of the library it calls."""
import ctypes
import os
import sys
import sysconfig

import numpy as np
import pytest

from paper_2512_24545_b200 import mdbf as M


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2512_24545_b200 import build
    build.build()


@pytest.fixture(params=["module", "ctypes"], autouse=True)
def way(request, monkeypatch):
    monkeypatch.setattr(M, "_calls", None)
    if request.param == "ctypes":
        monkeypatch.setattr(M, "CALLS_PATH", "/nonexistent")
    assert (M.calls() is M._CtypesCalls) == (request.param == "ctypes")
    return request.param


@pytest.mark.parametrize("handle", [0, None, ctypes.c_void_p(0), ctypes.c_void_p()])
@pytest.mark.parametrize("call", [M.mdbf_linear_forward, M.mdbf_linear_forward_host, M.mdbf_linear_forward_host_async])
def test_single_calls_refuse_a_null_handle(call, handle):
    x = np.zeros(4, dtype=np.float32)
    for buf in (x, x.ctypes.data, None):
        with pytest.raises(M.MdbfError) as e:
            call(handle, buf, y_host=x.ctypes.data, T=1, act_dtype=M.F32) if "host" in call.__name__ else call(handle, buf, y=x.ctypes.data, T=1, act_dtype=M.F32)
        assert e.value.status == M.ERR_INVALID_ARG


@pytest.mark.parametrize("n,status", [(0, M.ERR_SHAPE), (1, M.ERR_INVALID_ARG), (64, M.ERR_INVALID_ARG), (65, M.ERR_SHAPE), (1000, M.ERR_SHAPE)])
def test_lists_of_layers(n, status):
    for call in (lambda: M.mdbf_linear_forward_siblings([0] * n, 8, [8] * n, 1, M.BF16), lambda: M.mdbf_linear_forward_group([0] * n, [8] * n, (8,) * n, 1, M.BF16),
                 lambda: M.mdbf_linear_forward_sum([0] * n, 8, 8, 8, 1, M.BF16)):
        with pytest.raises(M.MdbfError) as e:
            call()
        assert e.value.status == status


def test_wrong_arguments_raise():
    with pytest.raises(ValueError):
        M.mdbf_linear_forward_siblings([8, 8], 8, [8], 1, M.BF16)       # fewer outputs than layers
    with pytest.raises(ValueError):
        M.mdbf_linear_forward(0, np.zeros((4, 4))[:, 1], 8, 1, M.F32)   # not contiguous
    with pytest.raises((TypeError, ctypes.ArgumentError)):
        M.mdbf_linear_forward(0, 8, 8, 1.5, M.F32)
    with pytest.raises(TypeError):
        M.mdbf_linear_forward_group(3, [8], [8], 1, M.F32)


def test_the_module_calls_the_library_it_was_given(way):
    """Not one it is linked to: the functions of whatever library ctypes has loaded (LIB_PATH), here of Python callbacks."""
    if way == "ctypes":
        pytest.skip("the module's own")
    vp, i32 = ctypes.c_void_p, ctypes.c_int32
    seen = []
    one = ctypes.CFUNCTYPE(i32, vp, vp, vp, i32, i32, vp)
    ptrs = ctypes.POINTER(vp)
    fns = [one(lambda *a, k=k: seen.append((k, a)) or k) for k in (11, 12, 13)]
    fns.append(ctypes.CFUNCTYPE(i32, ptrs, i32, vp, vp, vp, i32, i32, vp)(lambda hs, n, *a: seen.append((14, hs[:n], a)) or 14))
    fns.append(ctypes.CFUNCTYPE(i32, ptrs, i32, vp, ptrs, i32, i32, vp)(lambda hs, n, x, ys, *a: seen.append((15, hs[:n], x, ys[:n], a)) or 15))
    fns.append(ctypes.CFUNCTYPE(i32, ptrs, i32, ptrs, ptrs, i32, i32, vp)(lambda hs, n, xs, ys, *a: seen.append((16, hs[:n], xs[:n], ys[:n], a)) or 16))
    C = M.calls()
    try:
        C.set_library(M._addr, tuple(ctypes.cast(f, vp).value for f in fns))
        assert [f(1, 2, 3, 4, 5, 6) for f in (C.linear_forward, C.linear_forward_host, C.linear_forward_host_async)] == [11, 12, 13]
        assert C.linear_forward_sum([1, 2], 3, 4, 5, 6, 7, 8) == 14
        assert C.linear_forward_siblings((1, 2), 3, [4, 5], 6, 7, 8) == 15
        assert C.linear_forward_group([1], [2], [3], 4, 5, 6) == 16
        assert seen == [(k, (1, 2, 3, 4, 5, 6)) for k in (11, 12, 13)] + [(14, [1, 2], (3, 4, 5, 6, 7, 8)), (15, [1, 2], 3, [4, 5], (6, 7, 8)),
                                                                            (16, [1], [2], [3], (4, 5, 6))]
        with pytest.raises(ValueError):
            C.set_library(M._addr, (1, 2, 3, 4, 5, 0))
    finally:
        C.set_library(M._addr, tuple(ctypes.cast(getattr(M.lib(), name), vp).value for name in M._FORWARDS))


def test_the_module_belongs_to_one_interpreter_and_needs_not_be_there(way, monkeypatch, tmp_path, capsys):
    from paper_2512_24545_b200 import build
    assert build.CALLS == os.path.join(os.path.dirname(build.CALLS), "mdbf_calls" + sysconfig.get_config_var("EXT_SUFFIX"))
    assert sys.implementation.cache_tag.split("-")[1] in os.path.basename(build.CALLS)
    out = str(tmp_path / "m.so")
    monkeypatch.setenv("CC", "/nonexistent/cc")                   # no compiler: said, not raised
    assert build.build_calls(True, out) is False and not os.path.exists(out) and "ctypes" in capsys.readouterr().err
    monkeypatch.delenv("CC")
    assert build.build_calls(True, out) is True and os.path.exists(out)
