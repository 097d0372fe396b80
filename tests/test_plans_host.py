"""The host side's decisions (csrc/plans.h), compiled for the CPU."""
import ctypes
import os
import random
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
static int resident_of(int ks) { return ks == 1 ? 148 : 148 / ks * ks - 8 % ks; }
void t_plan_mat(int rows, int cols, int T, int kc, int nv, int *out) {
    plan_mat(rows, cols, T, kc, nv, resident_of, out, out + 1);
    out[2] = mt_tpr(out[0], out[1]);
    out[3] = mt_ring(kc, nv, out[0], 0);
    out[4] = (int)mt_smem_bytes(kc, nv, out[0], 0);
}
int t_small_ring(int kc, int nv, int bn, int ks) { return mt_ring(kc, nv, bn, (size_t)ks * plan_ceil_div(bn, ks) * MT_BM * 4); }
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


KC_NV = ((2, 4), (4, 3))                                         # chunks of the mode axis and V-image slots: l <= 16, l <= 32


@pytest.mark.parametrize("kc,nv", KC_NV)
def test_plan_of_the_large_token_tiles(plans, kc, nv):
    """Whatever the sizes: the ranks' sums of a split tile fit the activation ring they are pushed into, every rank has work, the tile is one
    the kernel takes, and its shared memory is what a CTA may have."""
    out = (ctypes.c_int * 5)()
    rng = random.Random(kc)
    log = lambda lo, hi: round(lo * (hi / lo) ** rng.random())
    split = 0
    for T in [*range(65, 1100), *(log(1100, 40000) for _ in range(200))]:
        for _ in range(100):
            rows, cols = log(1, 60000), log(1, 60000)
            plans.t_plan_mat(rows, cols, T, kc, nv, out)
            bn, ks, tpr, ring, smem = out
            case = (rows, cols, T, bn, ks, tpr, ring)
            assert 64 < bn <= 256 and bn % 16 == 0 and (bn >= T or bn % 64 == 0), case
            assert 1 <= ks <= 8 and 4 <= ring <= 12 and ring % 2 == 0 and smem <= 226 * 1024, case
            pairs = -(-(-(-cols // 64)) // 2)
            if ks > 1:
                split += 1
                assert -(-pairs // ks) * (ks - 1) < pairs, case
                assert tpr % 32 == 0 and tpr * ks >= bn, case
                assert ks * tpr * 128 * 4 <= ring * bn * 64 * 2, case
    assert split > 10000


@pytest.mark.parametrize("kc,nv", KC_NV)
def test_ring_of_the_small_token_tiles(plans, kc, nv):
    """Two or three buffers take turns at the ring: it has its full depth, a multiple of both, for every tile and split."""
    for bn in range(16, 65, 16):
        for ks in range(1, 9):
            assert plans.t_small_ring(kc, nv, bn, ks) == 12
