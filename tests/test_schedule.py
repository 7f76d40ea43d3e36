"""The closed form of the time-sliced schedule: every replica's steps are run
once and in order, by slots of equal shares, and the only wait of a slot is for
the first segment of the slot before it, which waits for nothing."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1207_2192_gb300", "csrc")
DRIVER = """
#include <cstdio>
#include <cstdlib>
#include "nd_schedule.h"
int main(int, char **v)
{
    const int B = atoi(v[1]), slots = atoi(v[3]);
    const long long n = atoll(v[2]), share = nd::slot_share(B, n, slots);
    nd::Segment g;
    for (int i = 0; i < slots + 2; ++i)
        for (int k = 0; k < nd::slot_segment(B, n, share, i, k, g); ++k)
            printf("%d %d %d %d %lld %lld\\n", i, g.pos, g.wait, g.signal, g.step_begin, g.nsteps);
}
"""


@pytest.fixture(scope="module")
def segments(tmp_path_factory):
    d = tmp_path_factory.mktemp("schedule")
    (d / "s.cpp").write_text(DRIVER)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", str(d / "s"), str(d / "s.cpp")], check=True)

    def run(B, n, slots):
        out = subprocess.run([str(d / "s"), str(B), str(n), str(slots)], check=True, capture_output=True, text=True).stdout
        return [tuple(map(int, l.split())) for l in out.splitlines()]
    return run


@pytest.mark.parametrize("B,n,slots", [
    (16, 2, 15), (16, 50, 15), (17, 3, 15), (30, 7, 15), (31, 5, 15), (47, 50, 15), (8, 2, 7), (15, 1000001, 7),
    (160, 4, 152), (256, 50, 152), (305, 2, 152), (153, 10 ** 10, 152), (1, 2, 2), (1, 7, 2), (64, 3, 63)])
def test_every_step_once_in_order_and_waits_that_end(segments, B, n, slots):
    segs = segments(B, n, slots)
    share = -(-B * n // slots)
    by_slot = [[s for s in segs if s[0] == i] for i in range(slots + 2)]
    assert max(len(sl) for sl in by_slot) <= B // slots + 2          # the room the table keeps for a slot
    assert not by_slot[slots] and not by_slot[slots + 1]
    done = sum(sum(s[5] for s in sl) for sl in by_slot)
    assert done == B * n and all(sum(s[5] for s in sl) <= share for sl in by_slot)
    for r in range(B):                                        # pieces follow one another from step 0 to n
        pieces = sorted((s for s in segs if s[1] == r), key=lambda s: s[4])
        at = 0
        for j, s in enumerate(pieces):
            assert s[4] == at and s[5] > 0
            at += s[5]
            assert s[2] == (j > 0) and s[3] == (j + 1 < len(pieces))
            if s[2]:                                          # what it waits for comes first in the slot before
                before = by_slot[s[0] - 1][0]
                assert before == pieces[j - 1] and not before[2]
        assert at == n and len(pieces) <= 2
