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


# Parameters that a kernel behind griddepcontrol.wait may hold as __restrict__:
# those it only writes, and those that no kernel before it in its chain writes.
_RESTRICT = {"k_adam": {"status", "half_copy"}, "k_arrange_weights": {"wfwd"}, "k_tc_weights": {"blob", "wfwd"},
             "k_forward_tc": {"table", "wblob", "status"}, "k_forward_tiny": {"grid4", "wblob", "status"}}


def _kernels(text):
    """(name, parameter list, body) of every __global__ function."""
    for m in re.finditer(r"__global__ void\s", text):
        at = m.end()
        while re.match(r"\s*__launch_bounds__\(", text[at:]):  # skip its balanced parentheses
            at = _close(text, text.index("(", at)) + 1
        open_ = text.index("(", at)
        close = _close(text, open_)
        body = text[close + 1:]
        if body.lstrip().startswith("{"):
            start = close + 1 + body.index("{")
            yield text[at:open_].split()[-1], text[open_ + 1:close], text[start:_close(text, start, "{", "}")]


def _close(text, at, a="(", b=")"):
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == a) - (text[i] == b)
        if depth == 0:
            return i
    raise AssertionError("unbalanced")


def test_dependents_read_through_plain_pointers():
    # What the predecessor of a programmatic dependent writes is read after
    # the wait through pointers without __restrict__, which would let the
    # compiler read it before.
    waits = set()
    for name, text in _sources().items():
        for kernel, params, body in _kernels(text):
            if "grid_dep_wait()" in body:
                waits.add(kernel)
                held = set(re.findall(r"__restrict__\s+(\w+)", params))
                assert held <= _RESTRICT.get(kernel, set()), (name, kernel, held)
    assert {"k_adam", "k_arrange_weights", "k_tc_weights", "k_forward_tc", "k_forward_tiny"} <= waits
