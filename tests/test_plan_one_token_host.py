"""The one-token kernel's split of the reduction (csrc/plans.h), compiled for the CPU."""
import ctypes
import os
import random
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_24545_b200", "csrc")
SHIM = """
#include "plans.h"
extern "C" int t_ranks(int n, const int *row_blocks, const int *pairs, int max_ks, int terms) { return mdbf::plan_t1_ranks(n, row_blocks, pairs, max_ks, terms); }
extern "C" int t_slots(int ks) { return mdbf::kT1Slots[ks]; }
"""


def test_ranks_of_one_token_launches(tmp_path):
    """No rank without work in any layer, a portable cluster for a sum's terms together, clusters that are whole, and a second wave only
    where it leaves a CTA less to do than one rank would."""
    (tmp_path / "shim.cpp").write_text(SHIM)
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-Werror", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(tmp_path / "p.so"), str(tmp_path / "shim.cpp")])
    L = ctypes.CDLL(str(tmp_path / "p.so"))
    assert all(L.t_slots(ks) <= 148 and L.t_slots(ks) // ks * ks == L.t_slots(ks) for ks in range(1, 9))
    rng = random.Random(4)
    seen = set()
    for _ in range(40000):
        n = rng.choice([1, 1, 2, 3, 4])
        terms = n if rng.random() < 0.2 else 1
        rb = [1 + int(2 ** rng.uniform(0, 9)) for _ in range(n)]
        pr = [max(1, int(2 ** rng.uniform(0, 8))) for _ in range(n)]
        ks = L.t_ranks(n, (ctypes.c_int * n)(*rb), (ctypes.c_int * n)(*pr), 8 // terms, terms)
        assert 1 <= ks and ks * terms <= 8
        assert all(-(-p // ks) * (ks - 1) < p for p in pr)
        if sum(rb) * ks > L.t_slots(ks * terms):
            assert ks == 1 or sum(rb) * ks <= 2 * L.t_slots(ks * terms) or -(-max(pr) // ks) + 24 < max(pr) + 24
        seen.add(ks)
    assert seen == set(range(1, 9))
