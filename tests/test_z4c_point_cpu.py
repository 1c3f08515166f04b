"""The Z4c right-hand side and constraints at one cell, compiled for the host,
against the same equations in 113-bit arithmetic: the integer sums may be no
less accurate than the FP64 form, whatever the components' sizes relative to
one another (z4c_point_check.cpp describes the states)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

CASES = ([("stretch", r, a) for r in (1.0, 4.0, 100.0, 1e4, 1e6) for a in (1.0, 0.01)] +
         [("offdiag", e, 1.0) for e in (1e-4, 1e-8, 1e-12)] + [("shift", e, 1.0) for e in (1e-4, 1e-8, 1e-12)] +
         [("plane", e, 0.1) for e in (1e-4, 1e-8)] +
         [(k, v, 1.0) for k in ("second", "first") for v in (float("inf"), float("nan"), 1e307, 1e150, 1e-310, 0.0)])
# what the integers leave to FP64: first derivatives that are no normal numbers, and results that are none
REFUSED = {float("inf"), 1e307, 1e-310}


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("point") / "z4c_point_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-w", "-I" + os.path.join(ROOT, "paper_2503_09629_gb300", "csrc"),
                    "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(cuda, "include"),
                    os.path.join(HERE, "z4c_point_check.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("kind,param,amp", CASES)
def test_integer_sums_as_accurate_as_fp64(program, kind, param, amp):
    """RMS error over RMS value of every right-hand side and constraint: at most
    1.25 times the FP64 form's (the integer sums round less often; both round
    the same FP64 remainder), itself a few roundings of 2^-53."""
    lines = subprocess.run([program, kind, repr(param), repr(amp)], check=True, capture_output=True,
                           text=True).stdout.splitlines()
    assert len(lines) == 31
    assert lines[30] == "finiteness differs 0"
    refused = kind == "first" and (param in REFUSED or param != param)
    assert (lines[29] != "refused 0") == refused
    for line in lines[:29]:
        f, fixed, fp64 = line.split()
        fixed, fp64 = float(fixed), float(fp64)
        if kind not in ("first", "second") or param == 0.0:
            assert fixed <= 1.25 * fp64 and fp64 <= 1e-15, (f, fixed, fp64)
