"""The kernels of a launch sequence run while the ones before still write the arena, so the
read-only path (`__ldg`, and const __restrict__ pointers, which the compiler may read through it)
is open to uploaded records alone, never to operands or bookkeeping."""
import glob
import os
import re

import paper_1807_02119_gb300 as pk

CSRC = os.path.join(os.path.dirname(pk.__file__), "csrc")
RECORDS = {"blob", "rec", "slots", "offs", "knots", "order", "leaves", "conv"}   # written by uploads only


def test_read_only_path_is_for_uploaded_records():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__ldg\(([^;]*);", code):
            assert re.match(r"\(const uint2\*\)\(blob \+", m.group(1)), (path, m.group(0))
            seen += 1
        for m in re.finditer(r"__restrict__\s+(\w+)", code):
            assert m.group(1) in RECORDS, (path, m.group(0))
            seen += 1
    assert seen >= 10
