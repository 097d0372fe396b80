"""Argument conversion of the forward calls' extension module, through calls that the library refuses before it touches a GPU."""
import ctypes

import numpy as np
import pytest

from paper_2512_24545_b200 import mdbf as M


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2512_24545_b200 import build
    build.build()


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
    with pytest.raises(TypeError):
        M.mdbf_linear_forward(0, 8, 8, 1.5, M.F32)
    with pytest.raises(TypeError):
        M.mdbf_linear_forward_group(3, [8], [8], 1, M.F32)
