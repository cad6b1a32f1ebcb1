"""The float-refined Stefan-Maxwell solve of the mixed unit and the block
fixed-point sums, compiled for the host, against 113-bit arithmetic.

Bounds: a velocity is the exact one to 2^-40 of the largest (the residual
in pairs of floats, 2^-46 of its terms, and the float correction), plus the
pairs of floats that hold j/rho and u (2^-46 of each), rounded to float once:
2^-24 |x| + 2^-40 max|x| + 2^-45 |u|.  1/tau_a is a product of pairs of
floats rounded once (2^-24; 1.001 allows for ties).  The error relative to
the largest velocity is on the whole no larger than that of the exact solution
rounded to float (0.1 %).  An absent species has velocity zero.  A sum of
eight products in limbs is rounded once (2^-53 of it), drops less than 2^-57
of the largest operand from each operand (half a unit of 2^-53 of it in
all), less than one unit of the sum per product (2^-56 of the largest operand
times the largest constant, one in all) and one unit at the end (an eighth)."""
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
    out = tmp_path_factory.mktemp("diffusion") / "diffusion_host"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", str(cuda), "-I", str(ROOT / "include"), "-o", str(out),
                    str(ROOT / "tests" / "diffusion_host.cpp"), "-lquadmath"] if os.uname().machine == "x86_64" else
                   ["true"], check=True)
    if not out.exists():
        pytest.skip("needs __float128")
    return out


@pytest.mark.parametrize("mode", [0, 1, 2, 3, 4])
def test_refined_solve_and_fixed_sums(program, mode):
    r = subprocess.run([str(program), str(mode), "4000", str(11 + mode)], capture_output=True, text=True)
    assert r.returncode == 0, r
    worst, tau, rms, wrong, sums = (float(v) for v in r.stdout.split())
    assert worst <= 1.0
    assert tau <= 1.001
    assert rms <= 1.001
    assert wrong == 0
    assert sums <= 1.0
