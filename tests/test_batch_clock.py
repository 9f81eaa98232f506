"""A batch's step clock on the device and the host's step, with launches whose wait gave up between the
others: both advance with every launch, so the entry of the pulse tables that a launch looks up is the one
that the host has filled.  The arithmetic is compiled for the host from the library's header."""
import os
import subprocess

import pytest

from paper_2312_10316_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "trtr_internal.cuh"
using namespace trtr;

int main() {
    // a clock outside the tables is reported and answered by an entry whose levels are all inside
    int bad = 0;
    for (int steps : {1, 2, 4})
        for (long long n = -200; n <= 200; ++n) {
            BatchClock c = {};
            c.n = n;
            c.first = 3;
            bool outside;
            const int e = c.table_entry(steps, &outside);
            bad += e < 0 || e + steps > kPulseLevels - 1;
            bad += outside == levels_within(c.first, (long)n, steps);
            bad += !outside && e != n - 1 - c.first;
        }
    // 10 000 launches of 1, 2 or 4 steps; the tables are filled from the host's step where they end
    unsigned r = 12345u;
    BatchClock c = {};
    long step = 0;
    bool ready = false;
    for (int k = 0; k < 10000; ++k) {
        r = r * 1664525u + 1013904223u;
        const int steps = 1 << ((r >> 16) % 3);
        if (!(ready && levels_within((long)c.first, step, steps))) {
            c.first = step - 1;
            ready = true;
        }
        bool outside;
        const int e = c.table_entry(steps, &outside);
        bad += outside || c.first + e != step - 1;
        c.n += steps;  // void or not (advance_clock)
        step += steps;
    }
    std::printf("%d\n", bad);
    return bad != 0;
}
"""


def test_launches_find_the_levels_that_the_host_has_filled(tmp_path):
    src = tmp_path / "clock.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "clock"
    subprocess.run([build.nvcc(), *build.NVCC_FLAGS, str(src), "-o", str(exe)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_blocks_that_gave_up_advance_the_clock_by_their_steps():
    """Read from the sources: every kernel that moves a batch's clock moves it through advance_clock, by the
    launch's steps on both ways out, and looks its tables up through table_entry_at alone."""
    text = {f: open(os.path.join(build.CSRC, f)).read() for f in ("trtr_batch.cu", "trtr_sweep.cu")}
    batch, sweep = text["trtr_batch.cu"], text["trtr_sweep.cu"]
    assert batch.count("advance_clock(clk, 1)") == 3 and batch.count("advance_clock(clk, 2)") == 2
    assert sweep.count("advance_clock(p.clk, kT)") == 1 and "advance_clock(p.clk, ok" not in sweep
    for t in text.values():
        assert "clk->done" not in t
    assert batch.count("table_entry_at(clk, 1,") == 1 and batch.count("table_entry_at(clk, 2,") == 1
    assert sweep.count("table_entry_at(p.clk, kT,") == 1
