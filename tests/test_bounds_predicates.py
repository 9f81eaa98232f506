"""The predicates of the bounds-checked build (CPU, compiled from the library's header): a plane's frame and
the pulse tables' entries, at their edges and against the index that a kernel would form."""
import subprocess

from paper_2312_10316_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "trtr_internal.cuh"
using namespace trtr;

static PlaneLayout layout(int nx, int ny, int gx, int gy) {
    PlaneLayout L;
    L.nx = nx;
    L.ny = ny;
    L.gx = gx;
    L.gy = gy;
    L.pitch = (nx + 2 * gx + gx - 1) / gx * gx;
    L.rows = ny + 2 * gy;
    L.plane = (size_t)L.rows * L.pitch;
    return L;
}

int main() {
    int bad = 0;
    for (int nx : {1, 16, 33, 130})
        for (int ny : {1, 32, 47})
            for (int w : {0, 1, 2, 4}) {
                const PlaneLayout L = layout(nx, ny, 32, 2);
                for (int j = -6; j < ny + 6; ++j)
                    for (int i = -70; i < nx + 70; ++i) {
                        const int wy = w < 2 ? w : 2;
                        const bool in = i >= -w && i < nx + w && j >= -wy && j < ny + wy;
                        bad += L.covers(i, j, w, wy) != in;
                        if (in) bad += L.at_w(i, j, L.gy) >= L.plane;
                    }
                // a frame wider than the allocation's: never outside it
                for (int i = -70; i < nx + 70; ++i)
                    if (L.covers(i, ny + 1, 1000, 1000)) bad += i + L.gx < 0 || i + L.gx >= L.pitch;
                bad += L.covers(0, ny + 2, 1000, 1000) || L.covers(0, -3, 1000, 1000);
                // tables: coordinate 0 of a level lies kTabGhost values behind its start
                const PulseTab t = PulseTab::make(nx, ny);
                for (int i = -12; i < nx + 160; ++i) {
                    const bool in = kTabGhost + i >= 0 && kTabGhost + i + 2 <= t.p2;
                    bad += t.covers(i, 2, 0) != in;
                }
                for (int j = -12; j < ny + 160; ++j) {
                    const int at = kTabGhost + t.y + 2 * j;  // of (Q1, Q2)
                    bad += t.covers(0, 2, j) != (at >= 2 * t.p2 && at + 2 <= t.level);
                }
            }
    std::printf("%d\n", bad);
    return bad != 0;
}
"""


def test_predicates_at_the_edges(tmp_path):
    src = tmp_path / "bounds.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "bounds"
    subprocess.run([build.nvcc(), *build.NVCC_FLAGS, "-DTRTR_BOUNDS_CHECK=1", str(src), "-o", str(exe)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
