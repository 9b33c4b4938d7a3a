"""Launch sizes that a call chooses by its shape (csrc/launch_rules.h), on the CPU."""
import ctypes
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_15619_b200", "csrc")

SOURCE = r"""
#include "launch_rules.h"
extern "C" int two_softmax(int T_q, int T_kv, int l) { return moda::fwd_two_softmax(T_q, T_kv, l); }
extern "C" int alternates(int d, int T, int G) { return moda::bwd_alternates(d, T, G); }
extern "C" unsigned row_ctas(int d, int bh, int T, int l, unsigned units, unsigned sms, int fp8) { return moda::bwd_row_ctas(d, bh, T, l, units, sms, fp8 != 0); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", "-o", str(d / "rules.so"), str(d / "rules.cpp")], check=True)
    return ctypes.CDLL(str(d / "rules.so"))


def _units(d, bh, T):
    return -(-bh * -(-T // 128) // (128 // d))


# B x heads, T, d, l, e4m3: SMs that were the best, or within 2 % of it, of the measured counts
BEST = [(128, 100, 64, 6, 0, 64), (128, 500, 64, 12, 0, 86), (64, 1024, 64, 12, 1, 86), (32, 2048, 64, 16, 1, 86),
        (128, 300, 128, 6, 0, 78), (128, 500, 128, 6, 0, 74), (64, 1024, 128, 30, 1, 128), (32, 8192, 128, 16, 0, 40), (64, 4096, 128, 23, 0, 72),
        (32, 5000, 128, 23, 1, 70), (32, 32768, 64, 32, 0, 22), (16, 65536, 64, 60, 0, 20), (16, 65536, 128, 24, 0, 16)]


@pytest.mark.parametrize("bh,T,d,l,fp8,best", BEST)
def test_sms_of_the_depth_part_where_they_were_measured(rules, bh, T, d, l, fp8, best):
    assert rules.row_ctas(d, bh, T, l, _units(d, bh, T), 148, fp8) == best


def test_sms_of_the_depth_part_over_all_shapes(rules):
    """As many as there are at most; even, or all units; fewer than 16 only at no more units for the busiest SM than 16 would leave it."""
    rng = random.Random(7)
    for _ in range(20000):
        d, fp8, sms = rng.choice((64, 128)), rng.randint(0, 1), rng.choice((148, 132, 16))
        bh, T, l = rng.randint(1, 256), int(2 ** rng.uniform(0, 17)), rng.randint(1, 256)
        units = _units(d, bh, T)
        n = rules.row_ctas(d, bh, T, l, units, sms, fp8)
        case = (d, bh, T, l, sms, fp8, units, n)
        assert 1 <= n <= min(units, sms), case
        assert n % 2 == 0 or n == units, case
        assert n >= min(16, units) or -(-units // n) == -(-units // 16), case


def test_alternate_iterations_where_they_were_measured_to_win(rules):
    assert not any(rules.alternates(128, T, G) for T in (1, 65536) for G in (1, 8))
    for T, G in ((1, 1), (512, 1), (768, 1), (128, 3), (256, 2)):
        assert not rules.alternates(64, T, G)
    for T, G in ((769, 1), (65536, 1), (129, 3), (257, 2), (300, 4), (100, 8)):
        assert rules.alternates(64, T, G)


def test_two_softmax_warpgroups_where_they_were_measured_to_win(rules):
    for T, l in ((129, 0), (129, 1), (256, 1), (257, 2), (512, 2), (2048, 4), (4096, 8), (8192, 16), (16384, 24)):
        assert rules.two_softmax(T, T, l), (T, l)
    for T, l in ((1, 0), (128, 0), (128, 1), (129, 2), (256, 2), (512, 4), (1000, 8), (4096, 16), (8192, 24)):
        assert not rules.two_softmax(T, T, l), (T, l)
    assert rules.two_softmax(2000, 15000, 24) and rules.two_softmax(1, 100, 0) and rules.two_softmax(1, 65536, 24) and not rules.two_softmax(64, 96, 1)
