"""The index checks of the KIN_DEBUG build at the launch shapes that the library
chooses itself (tests/debug_build_shapes.py): every check passes, parity with the
FP64 oracle holds, no guard byte changes.

Bounds: one step's parity tolerance of the storage type for each step taken (a
step adds at most its own), and the tolerance of E on a given state.
"""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
TOL = {3: 1e-12, 0: 1e-5, 1: 2e-3, 2: 1.6e-2}  # keyed by storage code
TOL_E = {3: 1e-12, 0: 2e-6, 1: 2e-6, 2: 2e-6}


def test_debug_build_at_the_chosen_shapes():
    r = subprocess.run([sys.executable, os.path.join(HERE, "debug_build_shapes.py")], capture_output=True, text=True,
                       timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    res = json.loads(r.stdout.strip().splitlines()[-1])
    assert res["debug_build"] is True
    assert len(res["cases"]) > 35
    for c in res["cases"]:
        assert c["debug_word"] == 0, c
        assert c["guards"] == "ok", c
        assert c["err"] < TOL[c["storage"]] * c["steps"], c
        assert c["err_E"] < TOL_E[c["storage"]], c
