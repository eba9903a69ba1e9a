"""The limits of the bounded device waits (csrc/bh_wait.h) on given clock readings."""
import os
import subprocess

SRC = r"""
#include <cstdio>
#include "bh_wait.h"
// polls of a wait that nothing satisfies, the clock read at every 64th; step(i): nanoseconds since the reading before
template <class F>
static long long polls(F step)
{
    unsigned long long now = 12345678901234ull;
    bh::WaitLimit lim(now);
    long long n = 0;
    for (int i = 0; i < lim.end; i++, n++)
        if ((i & 63) == 63) lim.look(i, now += step(i / 64));
    return n;
}
int main()
{
    const unsigned long long us = 1000ull, ms = 1000 * us, s = 1000 * ms;
    const long long more = 65536, most = 1 << 22;
    // a stop of 3 s, or of an hour, leaves that many polls
    printf("%d\n", polls([&](int i) { return i == 5 ? 3 * s : us; }) >= more);
    printf("%d\n", polls([&](int i) { return i == 0 ? 3600 * s : us; }) >= more);
    // so do time slices, off the GPU for 200 ms after every 640 polls
    printf("%d\n", polls([&](int i) { return i % 10 == 9 ? 200 * ms : us; }) >= more);
    // 64 polls take 100 us: over 65536 polls after a second, and at once no more
    const long long n = polls([&](int) { return 100 * us; });
    printf("%d\n", n >= 640000 + more && n <= 640000 + more + 130);
    // no more than 2^22 polls whatever the clock
    printf("%d\n", polls([&](int) { return us; }) == most && polls([&](int i) { return i == 65535 ? 2 * s : us; }) == most);
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
