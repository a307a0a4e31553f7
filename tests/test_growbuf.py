"""Growing scratch buffers (csrc/growbuf.h, host code): compiled on its own with
the host compiler and an allocator that counts, checked without a GPU.

* a buffer that was handed out is never freed by growing (a batch's tables and
  captured graphs hold its address);
* what is retired stays within twice the present buffer, however slowly the
  needs grow;
* a failed allocation frees what the attempt had allocated and changes nothing;

and the sources grow scratch in no other way."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2509_24236_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <set>
#include "growbuf.h"
std::set<void*> live;
long long left = -1;  // allocations before one fails; < 0: none does
int freed = 0;
int alloc(void** p, size_t bytes, bool zero) {
    if (left == 0) return 2;
    if (left > 0) --left;
    *p = zero ? std::calloc(1, bytes) : std::malloc(bytes);
    live.insert(*p);
    return 0;
}
void release(void* p) { live.erase(p); ++freed; std::free(p); }
int main() {
    std::vector<void*> retired;
    float* a = nullptr;
    int* b = nullptr;
    auto grow = [&](long long n) {
        return pf::grow_all(retired, {{&a, size_t(n) * sizeof(float), false}, {&b, size_t(n) * sizeof(int), true}}, alloc, release);
    };
    long long cap = 0, kept = 0, n_kept = 0;
    for (long long need = 1; need < 3000; need += 1 + need % 3) {
        if (need <= cap) continue;
        const long long to = pf::grown_capacity(cap, need);
        if (to < need || grow(to) != 0) return 1;
        kept += cap;
        n_kept += cap > 0 ? 2 : 0;
        cap = to;
        for (long long i = 0; i < cap; ++i) if (b[i] != 0) return 2;
        for (long long i = 0; i < cap; ++i) { a[i] = 1.0f; b[i] = 7; }
        if (kept > 2 * cap) return 3;
        if ((long long)retired.size() != n_kept || freed != 0) return 4;
        for (void* p : retired) if (!live.count(p)) return 5;
    }
    if (pf::grown_capacity(100, 100) != 100 || pf::grown_capacity(100, 101) != 150 || pf::grown_capacity(100, 900) != 900) return 6;
    float* const a0 = a;
    int* const b0 = b;
    left = 1;  // the first buffer is there, the second is refused
    if (grow(2 * cap) != 2 || a != a0 || b != b0 || freed != 1 || (long long)retired.size() != n_kept) return 7;
    std::printf("ok\n");
    return 0;
}
"""


def test_growth_keeps_what_was_handed_out(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    (tmp_path / "h.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, str(tmp_path / "h.cpp"), "-o", str(tmp_path / "h")], check=True)
    r = subprocess.run([str(tmp_path / "h")], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout == "ok\n", r.returncode


def test_a_call_on_a_live_volume_frees_no_scratch():
    """cudaFree stands only where a volume, a batch or a failed creation ends
    (and where new buffers of a failed growth are given back)."""
    allowed = {"pf_create_volume", "pf_destroy_volume", "pf_batch_destroy", "align_release", "free_list", "grow_scratch"}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"\bcudaFree\(", text):
            # the last definition that starts in column 0 before it
            head = re.findall(r"^(?!static_assert)[a-z][^\n;{}]*?\b(\w+)\([^;{}]*\)\s*\{", text[:m.start()], re.M)
            assert head and head[-1] in allowed, (os.path.basename(path), head[-1:])
