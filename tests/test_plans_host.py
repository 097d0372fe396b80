"""The host side's decisions (csrc/plans.h), compiled for the CPU."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_24545_b200", "csrc")
SHIM = r"""
#include "plans.h"
using namespace mdbf;
extern "C" {
uint64_t t_host_view(int pinned, uint64_t device, uint64_t start, size_t size, size_t bytes) {
    return host_view(HostRange{pinned != 0, device, start, size}, bytes);
}
int t_host_store_direct(uint64_t device, size_t es, int T) { return host_store_direct(device, es, T); }
int t_orth_ctas(int n, int chunk, int most, int sms) { return orth_ctas(n, chunk, most, sms); }
}
"""


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    d = tmp_path_factory.mktemp("plans")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-Werror", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "plans.so"), str(d / "shim.cpp")])
    L = ctypes.CDLL(str(d / "plans.so"))
    u64, sz = ctypes.c_uint64, ctypes.c_size_t
    L.t_host_view.argtypes, L.t_host_view.restype = [ctypes.c_int, u64, u64, sz, sz], u64
    L.t_host_store_direct.argtypes = [u64, sz, ctypes.c_int]
    return L


@pytest.mark.parametrize("pinned,off,size,nbytes,ok", [
    (1, 0, 16384, 16384, True), (1, 100, 16384, 16284, True),        # all of it, up to the last byte
    (1, 0, 16384, 16385, False), (1, 100, 16384, 16285, False),      # one byte past the mapping
    (1, 8191, 8192, 22016, False),                                   # starts on its last byte: a registered part of a larger array
    (1, 8192, 8192, 1, False), (0, 0, 0, 1, False), (0, 0, 16384, 8, False), (1, 0, 0, 1, False)])
def test_a_host_buffer_has_to_lie_in_one_pinned_mapping(plans, pinned, off, size, nbytes, ok):
    start = 0x7F0000000000
    assert plans.t_host_view(pinned, start + off, start, size, nbytes) == (start + off if ok else 0)
    assert plans.t_host_view(pinned, 0, 0, size, nbytes) == 0        # no device address
    assert plans.t_host_view(pinned, start - 1, start, size, 1) == 0


@pytest.mark.parametrize("off,es,T,ok", [(0, 2, 1, 1), (2, 2, 64, 1), (1, 2, 1, 0), (16, 4, 8, 1), (4, 4, 1, 1), (2, 4, 1, 0), (3, 4, 1, 0),
                                         (0, 2, 65, 0), (0, 4, 2048, 0)])      # more than 64 tokens: stored through a tensor map
def test_which_y_the_kernels_store_themselves(plans, off, es, T, ok):
    assert plans.t_host_store_direct(0x7F0000000000 + off, es, T) == ok
    assert plans.t_host_store_direct(0, es, T) == 0


@pytest.mark.parametrize("sms", [1, 16, 32, 74, 128, 148])
@pytest.mark.parametrize("n", [1, 128, 129, 5000, 28672, 1 << 21])
def test_a_cooperative_launch_fits_on_the_device(plans, n, sms):
    ctas, chunks = plans.t_orth_ctas(n, 128, 128, sms), -(-n // 128)
    assert 1 <= ctas <= min(sms, 128, chunks)
    assert ctas == chunks or ctas == min(sms, 128)
