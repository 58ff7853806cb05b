"""Rules for the device code that every rank of a multi-process run loads."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_01184_gb300", "csrc")


def test_no_tma_load_is_multicast():
    """A TMA load into several CTAs' shared memory is for code that runs on one
    GPU alone; the library is loaded by every rank.  (An arrival that
    tcgen05.commit sends to both CTAs of a pair moves no data.)"""
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h"))):
        with open(path) as f:
            # adjacent string literals are one instruction
            text = re.sub(r'"\s*\n\s*"', "", f.read())
        for m in re.finditer(r"cp\.async\.bulk[^\"]*", text):
            if "multicast" in m.group(0):
                found.append((os.path.basename(path), m.group(0)))
    assert not found
