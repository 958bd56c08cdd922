"""The lane arithmetic of groups of six lanes, run for a whole warp on the host:
every lane, the two that repeat lanes 24 and 25 among them, ends with the sums of
its own group, so that lanes which store the same entry store the same value."""
import os
import shutil
import subprocess

import pytest

import paper_2107_01104_gb300 as trk

CSRC = os.path.join(os.path.dirname(trk.__file__), "csrc")

PROGRAM = r"""
#include "six_lanes.h"
#include <cstdio>
using trk::SixLanes;
int main()
{
    // x[lane][k]: value k at the lane's column; lanes 30 and 31 hold what 24 and 25 hold
    double x[32][3], v[32], w[32];
    for (int l = 0; l < 32; ++l)
        for (int k = 0; k < 3; ++k) x[l][k] = 1 << (3 * SixLanes(l).u + k), x[l][k] += 1e7 * SixLanes(l).group;
    for (int l = 0; l < 32; ++l) {
        const SixLanes at(l);
        const int q = at.value(), p1 = at.partner(1) & 31, p2 = at.partner(2) & 31;   // (a shuffle's lane is taken mod 32)
        const double own = x[l][q], c1 = x[p1][SixLanes(p1).next(2)], c2 = x[p2][SixLanes(p2).next(1)];
        v[l] = ((q == 1 ? c1 : own) + (q == 2 ? c1 : c2)) + (q == 0 ? c1 : (q == 1 ? own : c2));
    }
    for (int l = 0; l < 32; ++l) w[l] = v[l] + v[l ^ 1];
    for (int l = 0; l < 32; ++l) {
        const int g = l < 30 ? l / 6 : 4;
        for (int k = 0; k < 3; ++k) {
            double want = 0;
            for (int u = 0; u < 6; ++u) want += (1 << (3 * u + k)) + 1e7 * g;
            const double got = w[SixLanes(l).holder(k) & 31];
            if (got != want) {
                std::printf("lane %d value %d: %.0f instead of %.0f\n", l, k, got, want);
                return 1;
            }
        }
    }
    return 0;
}
"""


def test_every_lane_has_its_own_groups_sums(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "lanes.cpp", tmp_path / "lanes"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
