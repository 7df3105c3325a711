"""The device waits' loops (fdtd_wait.h) on the host with a fake clock and a fake phase: the DFT kernel's wait gives up only
after a try made past its limit, so a block that was held up between a try and its look at the clock does not fail a
run whose copy is there."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_00234_gb300", "csrc")

PROGRAM = r"""
#include "fdtd_wait.h"
#include <cstdio>
struct World {
    unsigned long long t = 0, step, jump_at, jump, done_at;
    int tries = 0;
    bool done() { ++tries; return t >= done_at; }
    unsigned long long now() { t += t < jump_at && t + step >= jump_at ? jump : step; return t; }
};
int main()
{
    const unsigned long long never = ~0ull, limit = 1000;
    struct { World w; bool want; int most; } cases[] = {
        {{0, 10, never, 0, 0}, true, 1},              // complete before the first try
        {{0, 10, never, 0, 500}, true, 60},           // completes within the limit
        {{0, 10, never, 0, never}, false, 220},       // never completes: gives up soon after the second limit
        {{0, 10, 500, 100000, 600}, true, 60},        // held up past the limit; the phase completed meanwhile
        {{0, 10, 500, 100000, never}, false, 170},    // held up past the limit, never completes
        {{0, 5000, never, 0, 4000}, true, 5},         // every look at the clock takes longer than the limit
    };
    int q = 0;
    for (auto& c : cases) {
        const bool got = fdtd::patient_wait([&] { return c.w.done(); }, [&] { return c.w.now(); }, limit);
        if (got != c.want || c.w.tries > c.most) return std::printf("case %d: %d after %d tries\n", q, got, c.w.tries), 1;
        ++q;
    }
    return 0;
}
"""


def test_a_late_copy_is_no_failure(tmp_path):
    src = tmp_path / "wait.cpp"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(tmp_path / "wait")], check=True)
    r = subprocess.run([str(tmp_path / "wait")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
