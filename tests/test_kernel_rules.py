"""Rules of the CUDA sources that no run can show broken: what each kernel has
to do where a fault would need a wait that runs out in one warp alone."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_04315_gb300", "csrc")


def _sources():
    return {os.path.basename(p): open(p).read() for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*")))}


def test_every_warp_reports_its_own_timeout():
    # Every warp waits on its group's MMAs by itself, and after a group's last
    # tile no barrier passes a wait that gave up on to the others.
    found = 0
    for name, text in _sources().items():
        for m in re.finditer(r"atomicOr\(status, kStatusTimeout\)", text):
            line = text[text.rfind("\n", 0, m.start()) + 1:m.start()]
            assert "(t & 31) == 0" in line, (name, line.strip())
            found += 1
    assert found >= 3
