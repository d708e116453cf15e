"""How the solve server shares the GPU among a chunk's launches (csrc/deal.h), on the CPU: every launch that
has work gets some of it, whatever the mix and the GPU's size."""
import ctypes
import itertools
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHARE = [2, 1, 4, 2, 1]
TEAMS = [1, 2, 1, 1]


@pytest.fixture(scope="module")
def deal(tmp_path_factory):
    d = tmp_path_factory.mktemp("deal")
    (d / "t.cpp").write_text("""
#include "%s/paper_2302_07551_gb300/csrc/deal.h"
extern "C" void run(const int* n, const int* share, const int64_t* lv, const int* per, int per_sm, int sms, int cluster,
                    int slots, int32_t* clusters, int32_t* ctas) {
  mc::deal(mc::DealIn{5, 4, n, share, lv, per, per_sm, sms, cluster, slots}, clusters, ctas);
}
""" % ROOT)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-o", str(d / "t.so"), str(d / "t.cpp")])
    lib = ctypes.CDLL(str(d / "t.so"))

    def run(n, levels, sms, cluster, per_sm=2):
        out, ctas = (ctypes.c_int32 * 5)(), (ctypes.c_int32 * 4)()
        lib.run((ctypes.c_int * 5)(*n), (ctypes.c_int * 5)(*SHARE), (ctypes.c_int64 * 4)(*levels), (ctypes.c_int * 4)(*TEAMS),
                per_sm, sms, cluster, 8, out, ctas)
        return list(out), list(ctas)
    return run


@pytest.mark.parametrize("sms,cluster", [(152, 16), (132, 16), (64, 16), (60, 8), (16, 16), (8, 8)])
def test_every_launch_with_work_gets_a_part(deal, sms, cluster):
    for n in itertools.product([0, 1, 7, 200], repeat=5):
        for levels in [(0, 0, 0, 0), (0, 1, 0, 0), (0, 500, 3, 0), (0, 90000, 1, 7), (0, 0, 0, 512)]:
            clusters, ctas = deal(n, levels, sms, cluster)
            for g in range(5):
                assert (clusters[g] > 0) == (n[g] > 0) and clusters[g] <= n[g]
                assert clusters[g] <= 8 * SHARE[g]          # the launch's grid
            for c in range(4):
                assert (ctas[c] > 0) == (levels[c] > 0)
                assert ctas[c] <= -(-levels[c] // TEAMS[c])   # one team per level at most


def test_slots_follow_the_requests(deal):
    assert deal((0, 0, 0, 0, 3), (0, 0, 0, 0), 152, 16)[0] == [0, 0, 0, 0, 3]
    assert deal((200, 0, 0, 0, 0), (0, 0, 0, 0), 152, 16)[0] == [16, 0, 0, 0, 0]
    assert deal((200, 0, 0, 0, 0), (0, 600, 0, 0), 152, 16) == ([8, 0, 0, 0, 0], [0, 176, 0, 0])
    assert deal((0, 0, 40, 0, 1), (0, 0, 0, 0), 152, 16)[0] == [0, 0, 28, 0, 1]
