"""Read-only loads in programmatically launched kernels, by their source.

__ldg promises words that nothing writes while the grid lives.  A grid that
was launched programmatically lives while the kernel before it still runs, so
only tables, keys and masks, which are finished before a chain of kernels
starts, may be loaded that way: never a digit, a sum or a ciphertext."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_17341_gb300", "csrc")


def test_only_constants_are_loaded_read_only():
    found = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        assert "__restrict__" not in text and "ld.global.nc" not in text, path
        # kp: key words; w: twiddles (PassTw); ma.m1, ma.m2: the C^k masks
        for m in re.finditer(r"__ldg\(([^;\n]*)", text):
            found += 1
            assert re.match(r"(\(const ulonglong2 \*\)\()?(kp|w|ma\.m[12]\[ki\]) ", m.group(1)), (path, m.group(0))
    assert found >= 5
