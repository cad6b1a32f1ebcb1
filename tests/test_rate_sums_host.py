"""The sums of production rates in pairs of floats, compiled for the host,
against 113-bit arithmetic, for rates from cold gas (1e-47) to flames and for
densities of any unit.  Bounds: a term keeps 47 bits and adds 2^-48 of the sum
of rounding errors, the molar mass 47 bits: n 2^-45 of the largest of n terms,
then one rounding to float (2^-24), which may be to a subnormal (2^-149).  Sums
that do not cancel below 1/64 of their largest term are the nearest float
but for one in 2^45 / (64 n 2^24), 1300."""
import os
import shutil
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parents[1]
COUNT = 40000


@pytest.mark.parametrize("seed", [3, 5])
def test_pairs_of_floats(tmp_path, seed):
    cuda = Path(os.environ.get("CUDA_HOME", "/usr/local/cuda")) / "include"
    if shutil.which("g++") is None or not (cuda / "cuda_runtime.h").exists():
        pytest.skip("g++ and the CUDA headers are needed")
    if os.uname().machine != "x86_64":
        pytest.skip("needs __float128")
    out = tmp_path / "rate_sums_host"
    subprocess.run(["g++", "-O2", "-std=c++17", "-fno-strict-aliasing", "-I", str(cuda), "-I", str(ROOT / "include"),
                    "-o", str(out), str(ROOT / "tests" / "rate_sums_host.cpp"), "-lquadmath"], check=True)
    r = subprocess.run([str(out), str(COUNT), str(seed)], capture_output=True, text=True)
    assert r.returncode == 0, r
    worst, off = (float(v) for v in r.stdout.split())
    assert worst <= 1.0
    assert off <= COUNT / 1300
