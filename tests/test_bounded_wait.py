"""The bounded mbarrier wait of the tensor-core kernels (`mbar_wait` in tc_dev.cuh), its
source compiled for the host with a simulated barrier and clock: a pause of the whole
GPU (the clock jumps, the barrier completes meanwhile) does not end a wait, a barrier
that never completes does, after the time and the polls of its limit."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2408_04066_gb300", "csrc", "tc_dev.cuh")

HARNESS = r"""
#include <stdint.h>
#include <stdio.h>
#define __device__
#define __forceinline__ inline
%s
/* the barrier completes at time done_at; the GPU pauses for pause_ns right after poll number pause_after */
static uint64_t now, done_at, pause_ns;
static long polls, pause_after;
static uint64_t global_ns() { return now += 20; }
static bool mbar_try_wait(uint64_t*, uint32_t) {
    now += 100;
    const bool ok = now >= done_at;
    if (++polls == pause_after) now += pause_ns;
    return ok;
}
%s
static int run(uint64_t done, long after, uint64_t pause) {
    now = 1000; polls = 0; done_at = done; pause_after = after; pause_ns = pause;
    uint64_t bar = 0;
    return mbar_wait(&bar, 0) ? 1 : 0;
}
int main() {
    int bad = 0;
    bad |= !run(0, -1, 0);                                    /* complete at once */
    bad |= 2 * !run(5000, -1, 0);                             /* soon */
    for (long p = 1; p < 20000; p += p < 100 ? 1 : 997)       /* a pause after any poll, completed within it */
        bad |= 4 * !run(1000 + 130 * (uint64_t)p + 1000000, p, 3000000000ull);
    bad |= 8 * run(~0ull, -1, 0);                             /* never */
    bad |= 16 * (now < kTcWaitNs || now > 3 * kTcWaitNs);
    bad |= 32 * run(~0ull, 3, 3000000000ull);                 /* never, with a pause */
    bad |= 64 * (polls < 1000 || polls > 100000000);
    printf("%%d\n", bad);
    return 0;
}
"""


def test_bounded_wait(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    text = open(SRC).read()
    limits = "".join(re.findall(r"constexpr uint\d+_t kTcWait\w+ = [^\n]*\n", text))
    m = re.search(r"__device__ __forceinline__ bool mbar_wait\(.*?\n\}\n", text, re.S)
    assert m and limits
    c = tmp_path / "wait.cpp"
    c.write_text(HARNESS % (limits, m.group(0)))
    exe = tmp_path / "wait"
    subprocess.run([gxx, "-O1", "-std=c++17", str(c), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout
    assert int(out) == 0
