"""CPU checks that the sizes of workspaces follow the rules that choose the
kernels which use them."""
import ctypes as ct
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
    m x m matrices, four words, a flag per 256 entries), FP32 above m = 256 blocked (four padded
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
                need = max(need, 5 * m * m + 4 + (-(-m * m // 256) + 1) // 2)
        if m > 256:
            need = max(need, (4 * mp * mp + 1) // 2 + 1)
        assert have[m - 1] >= need, m


class _Stencil(ct.Structure):
    _fields_ = [("nx", ct.c_int), ("ny", ct.c_int), ("nz", ct.c_int),
                ("radius", ct.c_int), ("c1", ct.c_double), ("c2", ct.c_double),
                ("c1h", ct.c_float), ("c1l", ct.c_float), ("c2h", ct.c_float),
                ("c2l", ct.c_float)]


class _March(ct.Structure):
    _fields_ = [("tiles", ct.c_int), ("threads", ct.c_int), ("chunks", ct.c_int),
                ("zc", ct.c_int), ("pack", ct.c_int)]


def test_march_takes_every_point_once():
    """The geometry of the marching stencils (trm::zm_shape) and the place of a
    thread in it (zm_place, written out here): every group of every plane once,
    no more partial dots than the buffer holds, CTAs of at most 256 threads."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_1108_4509_gb300 as trm
    shape = ct.CDLL(trm.LIB_PATH)._ZN3trm8zm_shapeERKNS_9StencilOpEliii
    shape.restype = _March
    edges = [1, 2, 3, 5, 8, 9, 16, 33, 129]
    for nx in edges:
        for ny in edges:
            for nz in [1, 2, 5, 31, 70]:
                vw = 4 if nx % 4 == 0 else 2 if nx % 2 == 0 else 1
                N = nx * ny * nz
                dots = -(-(N // 4 if nx % 4 == 0 else N) // 256)
                for ncols in (1, 48):
                    z = shape(ct.byref(_Stencil(nx, ny, nz, 2)), ct.c_int64(N),
                              ncols, vw, dots)
                    nq = nx // vw * ny
                    assert z.threads % 32 == 0 and z.threads <= 256
                    assert z.tiles * z.chunks <= max(dots, z.tiles)
                    seen = []
                    for by in range(z.chunks):
                        for t in range(z.tiles * z.threads):
                            if z.pack == 1:
                                p, z0, on = t, by * z.zc, t < nq
                            else:
                                sub = t // nq
                                p, z0 = t - sub * nq, (by * z.pack + sub) * z.zc
                                on = sub < z.pack and z0 < nz
                            if on:
                                seen += [p * nz + k for k in
                                         range(z0, min(nz, z0 + z.zc))]
                    assert sorted(seen) == list(range(nq * nz)), (nx, ny, nz)
