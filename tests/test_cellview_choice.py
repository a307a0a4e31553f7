"""The choice of a volume's cell view (csrc/cellpitch.h, host code): compiled on
its own with the host compiler and checked without a GPU.

* padding rows and planes of records adds at most a sixteenth to the records of
  any grid;
* it decides no view away: a grid gets the view that unpadded records would
  get within the same budget, pitched when that fits too."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2509_24236_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include "cellpitch.h"
int main() {
    int nx, ny, nz;
    long long grid, narrow, wide, budget;
    while (std::scanf("%d %d %d %lld %lld %lld %lld", &nx, &ny, &nz, &grid, &narrow, &wide, &budget) == 7) {
        const pf::CellPitch p = pf::cell_pitch(nx, ny, nz);
        const pf::CellView v = pf::choose_view(nx, ny, nz, grid, narrow, wide, budget);
        std::printf("%lld %d %d %d %lld\n", p.count, v.mode, v.pitch.row, v.pitch.plane, v.pitch.count);
    }
    return 0;
}
"""

GRIDS = [(4, 4096, 4096), (4096, 4, 4096), (4096, 4096, 4), (4, 4, 4096), (5, 5, 900), (8, 8, 3000), (12, 40, 4096),
         (64, 64, 128), (512, 512, 1024), (33, 100, 100), (512, 512, 512), (2, 2, 2), (3, 4, 5)]


def old_choice(nodes, grid, narrow, wide, budget):
    """(mode) of unpadded records, one per node."""
    if grid + nodes * (narrow + wide) <= budget:
        return 1
    return 2 if wide and grid + nodes * narrow <= budget else -1


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("cellview")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(d / "h.cpp"), "-o", str(d / "h")], check=True)

    def ask(rows):
        inp = "".join(" ".join(str(v) for v in r) + "\n" for r in rows)
        out = subprocess.run([str(d / "h")], input=inp, capture_output=True, text=True, check=True).stdout
        return [tuple(int(v) for v in line.split()) for line in out.splitlines()]

    return ask


def test_padding_adds_at_most_a_sixteenth(choose):
    grids = [(a, b, c) for a in range(2, 70) for b in (2, 3, 4, 5, 8, 31, 64, 301) for c in (2, 4, 64, 1000)]
    for (nx, ny, nz), r in zip(grids, choose([(*g, 0, 8, 0, 0) for g in grids])):
        assert r[0] <= nx * ny * nz * 17 // 16, (nx, ny, nz)


@pytest.mark.parametrize("record", [(32, 0), (16, 32), (8, 32)])  # float, 16-bit, 8-bit grids
def test_the_view_is_that_of_unpadded_records(choose, record):
    narrow, wide = record
    rows, want = [], []
    for g in GRIDS:
        nodes = g[0] * g[1] * g[2]
        grid = 6 * nodes
        pitched = choose([(*g, 0, narrow, wide, 0)])[0][0]
        edges = [grid + n * r for n in (nodes, pitched) for r in (narrow, narrow + wide)]
        for budget in sorted({0, *edges, *(b - 1 for b in edges), 10 * edges[-1]}):
            rows.append((*g, grid, narrow, wide, budget))
            want.append(old_choice(nodes, grid, narrow, wide, budget))
    for row, mode, (pitched, got, r, p, count) in zip(rows, want, choose(rows)):
        assert got == mode, row
        if got > 0:
            need = narrow + (wide if got == 1 else 0)
            assert row[3] + count * need <= row[6]
            assert count == pitched or row[3] + pitched * need > row[6]
            assert count >= (row[0] - 2) + r * (row[1] - 2) + p * (row[2] - 2) + 1
