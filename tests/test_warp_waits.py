"""Waits made by whole warps end with one answer for the warp.  After a wait that
one lane's budget ended and another lane saw complete, the lanes would part
before the next warp collective (a shuffle, a tcgen05 load), which then waits for
good.  So in the kernels a plain mbar_wait belongs to single threads, which leave
by themselves, and whole warps use mbar_wait_warp or vote with warp_all (at once,
or, where nothing but plain reads lies between, at the next wait)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_29539_gb300", "csrc")
SINGLE = [r"if \((?:\w+ [=>] 0 \|\| |\w+ [=>]+ 0 && )?!\(ok = mbar_wait\(", r"bool ok = mbar_wait\(smem_u32\(&bar_a\)",
          r"\*ok = whole_warp \? mbar_wait_warp\(.*\) : mbar_wait\("]
VOTED = [r"__all_sync\(0xffffffffu, mbar_wait\(", r"warp_all\(mbar_wait\("]
LATER = [r"^ +mbar_wait\(.*\);  // \(if it gave up, so will the next wait\)$"]


def test_whole_warps_leave_together():
    plain = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        if os.path.basename(path) == "selftest.cu":  # its warp ends with the wait
            continue
        lines = open(path).read().splitlines()
        for n, line in enumerate(lines):
            if "mbar_wait(" not in line or any(re.search(p, line) for p in SINGLE + VOTED + LATER):
                continue
            if re.search(r"^ +ok = mbar_wait\(", line) and "ok = warp_all(ok);" in lines[n + 2]:
                continue
            plain.append(f"{os.path.basename(path)}:{n + 1}: {line.strip()}")
    assert not plain, plain
