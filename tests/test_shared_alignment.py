"""Dynamic shared memory lies behind a kernel's static arrays, so that its start is only as aligned as its declaration asks for; every one
of them is read in 16-byte words somewhere or may come to be, and says so."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_13089_b200", "csrc")


def test_dynamic_shared_arrays_declare_their_alignment():
    found = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for line in open(path):
            if re.match(r"\s*extern\s+__shared__", line):
                found += 1
                m = re.search(r"__align__\((\d+)\)", line)
                assert m and int(m.group(1)) % 16 == 0, "%s: %s" % (os.path.basename(path), line.strip())
    assert found >= 10
