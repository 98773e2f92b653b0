"""Kernel preparation (shared-memory limits, cluster sizes, occupancy) is shared by every thread that launches:
the library keeps what it has prepared in atomics, never in plain mutable statics.  No GPU: a data race
between two admission threads shows in no result here, so the sources are what is checked."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1608_00802_gb300", "csrc")


def test_no_plain_mutable_statics():
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.c*")) + glob.glob(os.path.join(CSRC, "*.h"))):
        for i, line in enumerate(open(path), 1):
            if re.match(r"\s*static\s+(bool|int|unsigned|uint32_t|size_t|long)\s+\w+\s*(\[|=|;)", line):
                found.append("%s:%d: %s" % (os.path.basename(path), i, line.strip()))
    assert not found, found
