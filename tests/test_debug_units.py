"""Every translation unit whose kernels check their indices hands its record to
kin_debug_status: a failed check skips the access, so one that nobody reads would
turn a wrong index into a silently wrong result."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1601_03815_gb300", "csrc")


def _text(path, seen):
    """The file's text with its quoted includes."""
    if path in seen or not os.path.exists(path) or os.path.basename(path) == "kin_debug.cuh":
        return ""
    seen.add(path)
    with open(path) as fh:
        own = fh.read()
    return own + "".join(_text(os.path.join(CSRC, name), seen) for name in re.findall(r'#include "([^"]+)"', own))


def test_every_unit_with_checks_is_read():
    with open(os.path.join(CSRC, "kin_api.cu")) as fh:
        api = fh.read()
    status = api[api.index("int kin_debug_status("):]
    checked = 0
    for unit in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        if "KIN_CHECK(" not in _text(unit, set()):
            continue
        checked += 1
        with open(unit) as fh:
            names = re.findall(r"^KIN_DEBUG_ACCESSOR\((\w+)\)", fh.read(), re.M)
        assert len(names) == 1, unit
        assert names[0] + "(" in status, (unit, names[0])
    assert checked >= 3
