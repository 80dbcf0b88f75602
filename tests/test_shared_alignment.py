"""Dynamic shared memory of the kernels (no GPU): its declared alignment is all
that the language promises of its first address, and the kernels read and write
it as double2, longlong2 and float4 (16 bytes)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2411_09605_gb300", "csrc")


def test_dynamic_shared_arrays_are_declared_16_byte_aligned():
    found, loose = 0, []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            for k, line in enumerate(f, 1):
                if re.search(r"\bextern\s+__shared__\b", line):
                    found += 1
                    if "__align__(16)" not in line:
                        loose.append(f"{os.path.basename(path)}:{k}")
    assert found > 0
    assert not loose, loose
