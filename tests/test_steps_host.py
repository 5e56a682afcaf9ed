"""Step counts against the step cap, up to the largest cap an int holds: the comparisons that the steppers make,
compiled for the host, against 64-bit arithmetic."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_13683_gb300", "csrc")

SOURCE = r"""
#include "fpt_steps.h"
#include <cstdio>
using namespace fpt_dev;

// A path that never passes, from group `grp` on: intervals of `groups` groups, the one with the cap step by step.
static int stepper(int grp, int groups, int nmax)
{
    for (int guard = 0; guard < 100000; ++guard) {
        if (!cap_inside(grp, groups, nmax)) {
            grp += groups;
            if (cap_reached(grp, nmax)) return steps_of(grp);
            continue;
        }
        for (int g = 0; g < groups; ++g, ++grp)
            for (int n = steps_of(grp), s = 0; s < 4; ++s)
                if (++n >= nmax) return n;
    }
    return -1;
}

int main()
{
    const int top = 2147483647;
    const int caps[] = {1, 2, 3, 4, 5, 7, 8, 4096, 4097, 5003, 1 << 24, 1 << 30, top - 4097, top - 5, top - 4,
                        top - 3, top - 2, top - 1, top};
    const int intervals[] = {1, 2, 8, 16, 32, 1024};
    for (int nmax : caps)
        for (int groups : intervals) {
            const long long last = nmax / 4, first = last > 2100 ? last - 2100 : 0;
            for (long long grp = first; grp <= last; ++grp) {
                const int g = (int)grp;
                bool ok = cap_inside(g, groups, nmax) == (4 * (grp + groups) > nmax) &&
                          cap_reached(g, nmax) == (4 * grp >= nmax) && cap_in_group(g, nmax) == (4 * grp + 4 >= nmax) &&
                          steps_of(g) == 4 * grp;
                for (int k = 0; k < 4; ++k) ok = ok && step_within(g, k, nmax) == (4 * grp + k + 1 <= nmax);
                if (!ok) { std::printf("cap %d, interval %d, group %lld\n", nmax, groups, grp); return 1; }
            }
            const int from = (int)(first - first % groups);
            if (stepper(from, groups, nmax) != nmax) { std::printf("cap %d, interval %d not reached\n", nmax, groups); return 1; }
        }
    return 0;
}
"""


def test_caps_are_reached_up_to_the_largest(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "steps.cpp", tmp_path / "steps"
    src.write_text(SOURCE)
    # signed overflow aborts
    subprocess.run([cxx, "-std=c++17", "-O1", "-ftrapv", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
