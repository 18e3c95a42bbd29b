"""CPU checks that the sizes of workspaces follow the rules that choose the
kernels which use them."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# trm::chol_work_elems by its mangled name
_PROBE = """
import ctypes as ct, sys
sys.path.insert(0, {root!r})
import __graft_entry__
__graft_entry__.build()
import paper_1108_4509_gb300 as trm
lib = ct.CDLL(trm.LIB_PATH)
have = lib._ZN3trm15chol_work_elemsEi
have.restype = ct.c_size_t
print([have(m) for m in range(1, 1025)])
"""


@pytest.mark.parametrize("blocked_from", [None, 33, 64, 128, 256, 257, 300, 4096])
def test_factorisation_workspace(blocked_from):
    """Every kernel that the rules let factor an m x m matrix finds its
    workspace, wherever TRM_CHOL_BLOCKED_FROM puts the line to the blocked
    launches: FP64 on one CTA (padded copy and a 33-row temporary) or blocked
    (four padded copies), the corrected FP32 factor for 33 <= m <= 256 (five
    m x m matrices, three deviations), FP32 above m = 256 blocked (four padded
    copies, in half as many doubles)."""
    env = dict(os.environ)
    env.pop("TRM_CHOL_BLOCKED_FROM", None)
    if blocked_from:
        env["TRM_CHOL_BLOCKED_FROM"] = str(blocked_from)
    r = subprocess.run([sys.executable, "-c", _PROBE.format(root=ROOT)],
                       capture_output=True, text=True, env=env, timeout=600)
    assert r.returncode == 0, r.stderr
    have = eval(r.stdout.strip().splitlines()[-1])
    line = blocked_from or 256
    for m in range(1, 1025):
        mp = -(-m // 32) * 32
        if m >= line:
            need = 4 * mp * mp + 1
        else:
            need = mp * (mp + 1) + 33 * mp
            if 33 <= m <= 256:
                need = max(need, 5 * m * m + 3)
        if m > 256:
            need = max(need, (4 * mp * mp + 1) // 2 + 1)
        assert have[m - 1] >= need, m
