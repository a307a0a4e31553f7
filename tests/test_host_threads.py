"""Different volumes may be used from different host threads, so no call keeps
a value in storage that all threads share without a lock: the library's sources
have no mutable function-local statics but the timing state (locked)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24236_gb300", "csrc")
LOCKED = {"static TimingState t;"}  # every use takes its mutex


def test_no_unlocked_function_local_statics():
    for path in sorted(glob.glob(os.path.join(CSRC, "*"))):
        if not path.endswith((".cu", ".cuh", ".h")):
            continue
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"^[ \t]+(static [^;({]*[;={])", text, re.M):
            line = m.group(1)
            if line in LOCKED or re.match(r"static (const|constexpr) ", line):
                continue
            raise AssertionError((os.path.basename(path), line))
