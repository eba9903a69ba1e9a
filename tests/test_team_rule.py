"""Which sets take the walk with a block of warps per group (bh_team_warps), on a GPU of 152 SMs, which have their
groups listed by cost (bh_groups_ordered), and which take the learned walk of four blocks per SM (bh_learned_four)."""
import os
import subprocess

import pytest

SRC = r"""
#include <cstdio>
#include "bh_internal.cuh"
using bh::WalkSet;
static WalkSet of(int systems, long long each, int G)
{
    return WalkSet((int)(systems * each), (int)each, systems * WalkSet::of_system(each, G));
}
static int batch(int systems, long long each, int G) { return bh::bh_team_warps(of(systems, each, G), G, 152); }
static int order(const WalkSet& s) { return bh::bh_groups_ordered(s); }
int main()
{
    // single systems: by the particles alone, at most 16 groups per SM
    for (int n : {1, 4096, 37000, 38000, 151000, 152000}) printf("%d ", bh::bh_team_warps(WalkSet(n, 96), 96, 152));
    printf("%d %d ", bh::bh_team_warps(WalkSet(1000, 128), 128, 152), bh::bh_team_warps(WalkSet(1000, 129), 129, 152));
    // a system is a group at least: thousands of small ones, and a few
    printf("%d %d %d %d ", batch(5000, 5, 96), batch(20000, 4, 64), batch(305, 1, 96), batch(304, 96, 96));
    // short walks: only while every group has a block at once
    printf("%d %d %d %d ", batch(256, 256, 64), batch(64, 256, 96), batch(32, 256, 96), batch(2, 512, 96));
    // middling ones: up to eight groups per SM
    printf("%d %d %d %d ", batch(64, 1024, 96), batch(128, 1024, 96), batch(32, 2047, 96), batch(64, 2047, 96));
    // long ones: as single systems, of which a batch of one is one
    printf("%d %d %d %d ", batch(16, 8192, 96), batch(4, 8192, 96), batch(100, 2048, 64), batch(1, 65536, 96));
    // by cost: single systems of more than 16384 and 200 G, short walks from 16 groups per SM on
    printf("%d %d %d %d ", order(WalkSet(16384, 32)), order(WalkSet(16385, 32)), order(WalkSet(19000, 96)), order(WalkSet(19500, 96)));
    printf("%d %d %d %d\n", order(of(512, 64, 64)), order(of(3000, 64, 64)), order(of(64, 1023, 96)), order(of(64, 1024, 96)));
    // 3648 groups
    printf("%d %d %d %d\n", bh::bh_learned_four(WalkSet(227000, 96), 96, 152), bh::bh_learned_four(WalkSet(228000, 96), 96, 152),
           bh::bh_learned_four(WalkSet(100000, 32), 32, 152), bh::bh_learned_four(WalkSet(1000, 128), 128, 152));
    return 0;
}
"""


def test_rule(tmp_path):
    from paper_1112_4539_gb300 import _build as b
    if not os.path.exists(b.NVCC):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "rule.cu", tmp_path / "rule"
    src.write_text(SRC)
    subprocess.run([b.NVCC] + b.ARCH + ["-std=c++17", "-I", b.CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert [int(v) for v in out] == [8, 8, 8, 4, 4, 0] + [8, 0] + [0, 0, 0, 8] + [0, 0, 8, 8] + [4, 0, 4, 0] + [4, 8, 0, 4] + [0, 1, 0, 1] + [0, 1, 0, 1] + [0, 1, 1, 1]
