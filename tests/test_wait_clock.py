"""The time limit of the bounded device waits (csrc/bh_wait.h) on given clock readings."""
import os
import subprocess

SRC = r"""
#include <cstdio>
#include "bh_wait.h"
using bh::WaitClock;
// readings until the wait is over, at most `most`; step(i): nanoseconds between readings i - 1 and i
template <class F>
static long long polls(F step, long long most)
{
    unsigned long long now = 12345678901234ull;
    WaitClock t(now);
    for (long long i = 1; i <= most; i++)
        if (t.over(now += step(i))) return i;
    return -1;
}
int main()
{
    const unsigned long long us = 1000ull, ms = 1000 * us, s = 1000 * ms;
    // one stop of 3 s, or of an hour, and then 900 ms of waiting
    printf("%d\n", polls([&](long long i) { return i == 5 ? 3 * s : us; }, 900000) == -1);
    printf("%d\n", polls([&](long long i) { return i == 1 ? 3600 * s : us; }, 900000) == -1);
    // time slices: off the GPU for 200 ms after each of 30 readings
    printf("%d\n", polls([&](long long i) { return i % 10 == 0 ? 200 * ms : us; }, 300) == -1);
    // a wait that nothing satisfies is over after a second
    const long long n = polls([&](long long) { return 10 * us; }, 10000000);
    printf("%d\n", n > 99990 && n < 100010);
    // and, whatever the readings, after a bounded number of long gaps
    printf("%d\n", polls([&](long long) { return 3600 * s; }, 1000) > 0);
    return 0;
}
"""


def test_stops_do_not_count_as_waiting(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    src, exe = tmp_path / "wait.cpp", tmp_path / "wait"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(root, "paper_1112_4539_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["1"] * 5
