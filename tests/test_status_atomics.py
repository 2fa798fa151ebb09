"""The step record's status word is shared by all warps of a launch, which raise its
bits with atomicOr: no kernel may write it with a plain store (a bit raised by a
warp that ran earlier would be lost).  Read from the sources: the order of such
a race cannot be forced.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_02125_gb300", "csrc")


def test_status_is_written_by_atomics_only():
    uses = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(path) as f:
            code = re.sub(r"//[^\n]*", "", f.read())
        uses += len(re.findall(r"atomic\w+\(&[\w.]+->status", code))
        plain = re.findall(r"->status\s*(?:[|&^+-]?=)(?!=)[^;]*;", code)
        assert not plain, (os.path.basename(path), plain)
    assert uses >= 3
