"""Asynchronous copies into shared memory, in the sources: the destination may
have been read just before (the gradient-row slots are, by the same thread), and
only a "memory" clobber keeps the compiler from moving those reads behind the
copy, or the reads of what it brings before the wait."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2603_05493_gb300", "csrc")


def test_every_cp_async_clobbers_memory():
    found, bare = 0, []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = open(path).read()
        for m in re.finditer(r"asm\s+volatile\s*\(\s*\"cp\.async\.(?:c[ag]|wait).*?\);", src, re.S):
            found += 1
            if '"memory"' not in m.group(0):
                bare.append("%s:%d" % (os.path.basename(path), src.count("\n", 0, m.start()) + 1))
    assert found >= 10
    assert not bare, bare
