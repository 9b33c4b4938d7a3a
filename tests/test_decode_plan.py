"""The cut of a decode step's key range into runs and pieces (csrc/decode_plan.h), on the CPU: every key of every group is in
exactly one piece, the pieces of a group are numbered in order and fit its partials, and what the merge kernel computes agrees."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_15619_b200", "csrc")

SOURCE = r"""
#include "decode_plan.h"
#include <vector>
using namespace moda;
// 0, or the line of the first condition that fails.  lens == nullptr: equal lengths.  out: aligned, longest run in units of keys
extern "C" int check(int B, int heads, int T_kv, const int* lens, int teams, int G, long long* out) {
#define NEED(c) do { if (!(c)) return __LINE__; } while (0)
    const int u = decode_unit_log2((long long)B * heads, T_kv), min_run = decode_min_run(T_kv, u);
    const int max_pieces = decode_units(T_kv, u) / min_run + 2 < kDecodeMaxSplits - 1 ? decode_units(T_kv, u) / min_run + 2 : kDecodeMaxSplits - 1;
    auto len = [&](int b) { return lens ? lens[b] : T_kv; };
    DecodeCut cut;
    if (!lens) {
        cut = decode_cut_equal(B * heads, T_kv, u, teams, G);
    } else {                                               // as the split kernel does it
        long long sum = 0;
        for (int b = 0; b < B; ++b) sum += decode_units(len(b), u);
        NEED(sum * heads < (1ll << 30));
        cut = DecodeCut{decode_run(int(sum) * heads, teams, min_run), 0};
        if (B * heads <= teams) {
            const int longer = decode_aligned_run(cut.run, 1), longest = decode_aligned_run(cut.run, G);
            auto pieces_of = [&](int run) { int n = 0; for (int b = 0; b < B; ++b) n += decode_ceil_div(decode_units(len(b), u), run); return n; };
            NEED(pieces_of(longer) < 65536 && pieces_of(longest) < 32768);
            if (B <= 32 && pieces_of(cut.run) * heads <= teams) cut.aligned = 1;
            else if (pieces_of(longer) * heads <= teams) cut = DecodeCut{longer, 1};
            else if (pieces_of(longest) * heads <= teams) cut = DecodeCut{longest, 1};
        }
    }
    std::vector<int> before(B + 1, 0);
    for (int b = 0; b < B; ++b) {
        const long long next = (long long)before[b] + DecodeWalk::stride_of(decode_units(len(b), u), cut);
        NEED(next * heads < (1ll << 31) - (1ll << 29));
        before[b + 1] = int(next);
    }
    const int total = before[B] * heads;
    NEED((long long)cut.run * teams >= total && (long long)cut.run * teams < (1ll << 31));
    std::vector<int> done((size_t)B * heads, 0), count((size_t)B * heads, 0), pieces((size_t)B * heads, 0);
    int b0 = 0;
    for (int team = 0; team < teams; ++team) {
        const long long first = (long long)team * cut.run;
        while (b0 + 1 < B && first >= (long long)before[b0 + 1] * heads) ++b0;
        DecodeWalk k;
        k.begin(cut, team, total, heads, u, b0, before[b0], len);
        int n = 0;
        for (; !k.done(); k.next(cut, heads, u, len)) {
            const DecodePiece w = k.piece(cut, team, u, len);
            NEED(w.b >= 0 && w.b < B && w.head_team >= 0 && w.head_team < heads);
            const size_t g = (size_t)w.b * heads + w.head_team;
            NEED(w.k_begin == done[g] && w.k_end > w.k_begin && w.k_end <= len(w.b));
            NEED(w.k_begin % kDecodeStageKeys == 0);
            NEED(w.index == count[g] && w.index < w.pieces && w.pieces <= max_pieces);
            NEED(count[g] == 0 || w.pieces == pieces[g]);
            pieces[g] = w.pieces;
            done[g] = w.k_end;
            ++count[g];
            ++n;
            NEED(((w.k_end - w.k_begin - 1) >> u) < cut.run);
        }
        NEED(!cut.aligned || n <= 1);
    }
    for (int b = 0; b < B; ++b)
        for (int h = 0; h < heads; ++h) {
            const size_t g = (size_t)b * heads + h;
            NEED(done[g] == len(b) && count[g] == pieces[g]);
            NEED(lens || pieces[g] == decode_pieces_equal(cut, int(g), T_kv, u));
        }
    out[0] = cut.aligned; out[1] = cut.run; out[2] = u;
    return 0;
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "plan.so"), str(d / "plan.cpp")], check=True)
    lib = ctypes.CDLL(str(d / "plan.so"))
    lib.check.argtypes = [ctypes.c_int] * 3 + [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_void_p]

    def check(B, heads, T_kv, lens, teams, G=1):
        out = np.zeros(3, dtype=np.int64)
        if lens is not None:
            lens = np.ascontiguousarray(lens, dtype=np.int32)
        rc = lib.check(B, heads, T_kv, None if lens is None else lens.ctypes.data, teams, G, out.ctypes.data)
        assert rc == 0, (B, heads, T_kv, teams, "condition in line", rc)
        return out
    return check


TEAMS = (148, 74, 37, 29, 24, 18, 12, 9)


@pytest.mark.parametrize("teams", TEAMS)
def test_equal_lengths(plan, teams):
    for B, heads in ((1, 1), (1, 2), (3, 1), (5, 3), (8, 1), (32, 1), (32, 3), (128, 1), (300, 2)):
        for T in (1, 63, 64, 65, 255, 256, 300, 1000, 4096, 8191, 8192, 40000, 131072, 1000001):
            plan(B, heads, T, None, teams)
            plan(B, heads, T, None, teams, G=8)


@pytest.mark.parametrize("teams", TEAMS)
def test_lengths_per_sequence(plan, teams):
    rng = np.random.default_rng(teams)
    for B, heads in ((1, 1), (1, 2), (2, 1), (7, 1), (8, 2), (32, 1), (33, 1), (40, 1), (130, 1), (288, 1), (300, 2), (620, 1)):
        for T in (1, 64, 200, 1000, 8192, 40000):
            for lens in (rng.integers(1, T + 1, size=B), np.ones(B), np.full(B, T), np.where(np.arange(B) == B // 2, T, 1)):
                plan(B, heads, T, lens, teams, G=8 if B % 2 else 4)


def test_a_piece_per_team_where_the_teams_suffice(plan):
    # 8 sequences of 4096 keys with 3 head teams each on 74 teams: three pieces of 22 stages; runs that cross the groups
    # would be 21 long and cost most teams two pieces
    aligned, run, _ = plan(8, 3, 4096, None, 74)
    assert aligned and run == 22
    aligned, run, _ = plan(8, 1, 4096, [64 * n for n in (9, 17, 64, 33, 5, 1, 50, 29)], 148)
    assert aligned and run in (4, 5)
    assert not plan(32, 1, 8192, [256 * (i + 1) for i in range(32)], 18)[0]


def test_counts_stay_inside_an_int(plan):
    """A block table may name the same page for every sequence, so the step's keys are not bounded by the cache's size."""
    for T in (1 << 20, 1 << 26, 2 ** 31 - 1):
        for B, heads in ((1, 1), (65535, 4), (65535, 16), (4096, 1)):
            out = plan(B, heads, T, None, 18)
            assert out[2] >= 6
            if B <= 4096:
                plan(B, heads, T, np.full(B, T), 148)
    assert plan(65535, 4, 1 << 26, np.full(65535, 1 << 26), 18)[2] > 6
