"""The cell view's pitch rule (csrc/cellpitch.h, host code): compiled on its
own with the host compiler and checked without a GPU.

* records of different cells never coincide and all lie inside the
  allocation (rows hold nx - 1 cells, planes ny - 1 rows, nz - 1 planes);
* neighbours along each axis, and diagonal ones along x-y and y-z, fall in
  different quarters of a 128-byte line of 32-byte records;
* a grid of equal sides needs no more records than it has nodes;
* the grids whose pitched view would pass 2^31 records keep the node pitch."""
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
    while (std::scanf("%d %d %d", &nx, &ny, &nz) == 3) {
        const pf::CellPitch p = pf::cell_pitch(nx, ny, nz);
        std::printf("%d %d %lld\n", p.row, p.plane, p.count);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def pitch(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("cellpitch")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(d / "h.cpp"), "-o", str(d / "h")], check=True)

    def ask(grids):
        inp = "".join("%d %d %d\n" % g for g in grids)
        out = subprocess.run([str(d / "h")], input=inp, capture_output=True, text=True, check=True).stdout
        return [tuple(int(v) for v in line.split()) for line in out.splitlines()]

    return ask


def test_records_are_distinct_inside_and_spread_over_the_quarters(pitch):
    sides = list(range(2, 40)) + [47, 48, 63, 64, 65, 100, 127, 128, 203, 251, 256, 384, 511, 512, 768, 1290]
    grids = [(n, n, n) for n in sides] + [(a, b, c) for a in (2, 3, 5, 64, 97) for b in (2, 7, 33) for c in (2, 50)]
    for (nx, ny, nz), (row, plane, count) in zip(grids, pitch(grids)):
        if (row, plane) == (nx, nx * ny):
            continue  # the node pitch: one record per node
        assert row >= nx - 1 and plane >= row * (ny - 1)
        last = (nx - 2) + row * (ny - 2) + plane * (nz - 2)
        assert nx * ny * nz <= count < 2 ** 31 and last < count
        assert row % 4 == 2 and plane % 4 == 3
        for step in (1, row, plane, 1 + row, 1 - row, row + plane, row - plane):
            assert step % 4 != 0
        if nx == ny == nz and nx >= 32:
            assert count == nx ** 3


def test_a_view_beyond_32_bit_records_keeps_the_node_pitch(pitch):
    wide, narrow = pitch([(128, 4096, 4095), (127, 4096, 4095)])  # 130 and 126 records a row
    assert wide == (128, 128 * 4096, 128 * 4096 * 4095)
    assert narrow[0] == 126 and narrow[2] < 2 ** 31
