"""What a waiting block concludes at a grid barrier (csrc/barrier.h), on the host.

Another block records an error and then arrives; every place of those two steps between
the waiting block's reads is tried.  A block that passes has to have seen an error recorded
before the last arrival.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "barrier.h"
#include <cstdio>
// The other block's steps: 1 records an error (if `fails`), 2 arrives.  Step k is made
// before the waiting block's read number at[k].
static int run(bool fails, int at1, int at2, uint64_t start)
{
    // three blocks, two have arrived
    gb::BarrierState b = gb::barrier_start(start, 3);
    b.target += 3;
    start += gb::barrier_arrival(false);
    uint64_t word = start + gb::barrier_arrival(false);
    int reads = 0, status = 0;
    auto others = [&] {
        if (at1 == reads && fails) status = -5;
        if (at2 == reads) word += gb::barrier_arrival(fails);
        ++reads;
    };
    for (int look = 0; look < 20; ++look) {
        const gb::BarrierLook l = gb::barrier_look(b, [&] { others(); return status; }, [&] { others(); return word; });
        if (l != gb::BARRIER_WAIT) return l;
    }
    return gb::BARRIER_WAIT;
}
int main()
{
    int bad = 0;
    // the words that a launch may start from: none, after other launches, errors among
    // them (their count about to wrap too), more arrivals than 32 bits hold
    const uint64_t starts[] = {0, 24, 24 + (uint64_t(5) << 48), (uint64_t(0xffff) << 48) + 3, 0xffffffffull,
                               uint64_t(3) * 0x55555556ull, uint64_t(3) << 40};
    for (uint64_t start : starts) {
        for (int a1 = 0; a1 < 12; ++a1)
            for (int a2 = a1; a2 < 12; ++a2) {
                bad += run(true, a1, a2, start) != gb::BARRIER_ERROR;
                bad += run(false, a1, a2, start) != gb::BARRIER_PASSED;
            }
        // an error and no arrival: the wait ends
        bad += run(true, 3, 1000, start) != gb::BARRIER_ERROR;
        bad += run(false, 3, 1000, start) != gb::BARRIER_WAIT;
    }
    std::printf("%d\n", bad);
    return bad != 0;
}
"""


def test_an_error_recorded_before_the_last_arrival_is_seen(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src = tmp_path / "look.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "look")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2012_13548_gb300", "csrc"), str(src),
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, "interleavings decided wrongly: " + r.stdout
