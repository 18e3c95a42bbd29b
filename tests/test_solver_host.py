"""The solver's host logic on the CPU: csrc/solver.cu as built, linked with the
fakes of tests/native/solver_fakes.cu instead of the CUDA runtime and the
kernels, so that a device wait that gives up, or a copy that the runtime
refuses, can be had without a GPU. What the fakes leave undefined becomes a
function that returns zero."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1108_4509_gb300", "csrc")
FAKES = os.path.join(ROOT, "tests", "native", "solver_fakes.cu")
CUDA = "/usr/local/cuda"


def _symbols(obj, kind):
    out = subprocess.run(["nm", obj], capture_output=True, text=True,
                         check=True).stdout
    return {ln.split()[-1] for ln in out.splitlines()
            if ln.split()[-2] in kind}


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    nvcc = shutil.which("nvcc") or os.path.join(CUDA, "bin", "nvcc")
    gxx, gcc = shutil.which("g++"), shutil.which("gcc")
    if not (os.path.exists(nvcc) and gxx and gcc and shutil.which("nm")):
        pytest.skip("needs nvcc, gcc and nm")
    import __graft_entry__
    __graft_entry__.build()
    tmp = tmp_path_factory.mktemp("solver_host")
    solver = os.path.join(ROOT, "paper_1108_4509_gb300", "_build", "solver.cu.o")
    fakes, stubs = str(tmp / "fakes.o"), str(tmp / "stubs.o")
    flags = ["-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17",
             "-I" + os.path.join(ROOT, "include"), "-I" + CSRC]
    subprocess.run([nvcc, *flags, "-c", FAKES, "-o", fakes], check=True)
    missing = (_symbols(solver, "U") | _symbols(fakes, "U"))
    missing -= _symbols(solver, "TWVBD") | _symbols(fakes, "TWVBD")
    missing = sorted(s for s in missing
                     if re.match(r"_?_?cuda|_ZNK?3trm", s))
    src = tmp / "stubs.c"
    src.write_text("".join(
        f'long f{i}(void) __asm__("{s}");\nlong f{i}(void) {{ return 0; }}\n'
        for i, s in enumerate(missing)))
    subprocess.run([gcc, "-O1", "-c", str(src), "-o", stubs], check=True)
    exe = str(tmp / "harness")
    subprocess.run([gxx, solver, fakes, stubs, "-lpthread", "-o", exe],
                   check=True)
    return exe


def _run(exe, what):
    r = subprocess.run([exe, what], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]


def test_every_timeout_reaches_the_caller(harness):
    """Whichever digit Gram of a solve gives up (the first orthonormalization,
    a phase change, an iteration, the closing step) the solve returns
    TRM_ETIMEOUT, trm_rayleigh_ritz likewise, and the next call starts clean."""
    _run(harness, "timeouts")


def test_host_blocks_with_columns_over_2_gb(harness):
    """trm_solve's C0 and C on the host, N % 4 != 0, N >= 2^28: the columns go
    one by one where a 2-D copy's pitch would not be accepted."""
    _run(harness, "large_columns")


def test_padding_cleared_where_the_generalized_ladder_turns_to_fp64(harness):
    """Full SP leaves FP32 entries where FP64 blocks have their padding rows:
    they are cleared before the first FP64 iteration."""
    _run(harness, "generalized")
