"""The float-refined Stefan-Maxwell solve of the mixed unit, compiled for the
host, for species far below the others: densities from the smallest subnormal
double to the normal floats (mode 0) and about the smallest float (3), and
one trace that alone moves, so that its momentum balances the others' (1);
and for another unit of density, 2^-70 to 2^70 times the first (2).
Every velocity is finite and the exact one to 2^-24 |x| (rounded to float
once) plus 2^-40 of the largest n_b |x_b| over the largest n_b (the residual
sums products n_b x_b in integers, 2^-53 of the largest, and takes its other
terms as pairs of floats, 2^-46 of each; the float correction adds 2^-22 of
itself) plus 2^-53 |u| (j - rho u is one operation in double)
plus 2^-100 (the floats' range)."""
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
    out = tmp_path_factory.mktemp("traces") / "diffusion_traces_host"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", str(cuda), "-I", str(ROOT / "include"), "-o", str(out),
                    str(ROOT / "tests" / "diffusion_traces_host.cpp"), "-lquadmath"], check=True)
    return out


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
def test_refined_solve_with_traces(program, mode):
    r = subprocess.run([str(program), str(mode), "4000", str(7 + mode)], capture_output=True, text=True)
    assert r.returncode == 0, r
    nonfinite, worst = (float(v) for v in r.stdout.split())
    assert nonfinite == 0
    assert worst <= 1.0
