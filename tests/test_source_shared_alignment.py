"""Dynamic shared memory is read and written 16 bytes at a time (tile products,
copies), so every kernel declares its buffer on a 16-byte boundary: an element
type of that alignment (double2, int4, ...) or an explicit one."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2304_01728_gb300", "csrc")


def test_dynamic_shared_buffers_are_16_byte_aligned():
    bad, seen = [], 0
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for i, line in enumerate(open(f), 1):
            m = re.search(r"extern __shared__ (.*?)\s+\w+\[\]", line)
            if not m:
                continue
            seen += 1
            a = re.search(r"__align__\((\d+)\)", m.group(1))
            if not (a and int(a.group(1)) >= 16) and m.group(1).split()[-1] not in ("double2", "int4", "uint4", "float4"):
                bad.append("%s:%d: %s" % (os.path.basename(f), i, line.strip()))
    assert seen > 10 and not bad, bad
