"""The sums over partner species of the double collision in 58-bit limbs,
compiled for the host, against 113-bit arithmetic: every species present (mode
0), heavy ones with traces of light ones (1), absent ones (2), in every
direction, at rest and moving.  Bound, in units of 2^-53 of the largest product
times the sum of the constants: a difference of two products has six
truncations of one unit (two factors, one partial product, twice), one of the
fold and half a unit of rounding, where the larger product is at least 2^56
units: 1.0.  The constants' truncation adds 1/8, their partial
products at most eight units of 2^55 over the sum of the constants: below 0.9.
So 2.0.  The root mean square error is no larger than that of the floating
form, and differences that vanish give zero."""
import os
import shutil
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parents[1]


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cuda = Path(os.environ.get("CUDA_HOME", "/usr/local/cuda")) / "include"
    if shutil.which("g++") is None or not (cuda / "cuda_runtime.h").exists():
        pytest.skip("g++ and the CUDA headers are needed")
    if os.uname().machine != "x86_64":
        pytest.skip("needs __float128")
    out = tmp_path_factory.mktemp("limbs") / "limb_differences_host"
    subprocess.run(["g++", "-O2", "-std=c++17", "-fno-strict-aliasing", "-I", str(cuda), "-I", str(ROOT / "include"),
                    "-o", str(out), str(ROOT / "tests" / "limb_differences_host.cpp"), "-lquadmath"], check=True)
    return out


@pytest.mark.parametrize("mode", [0, 1, 2])
def test_limb_differences(program, mode):
    r = subprocess.run([str(program), str(mode), "20000", str(11 + mode)], capture_output=True, text=True)
    assert r.returncode == 0, r
    worst, rms, floating, off = (float(v) for v in r.stdout.split())
    assert worst <= 2.0
    assert rms <= floating
    assert off == 0
