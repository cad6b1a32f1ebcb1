"""The autotuner tries the choice by the lattice's size that an untuned context
has, and keeps it (0) unless a fixed block size is faster by more than the
timings differ."""
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
    out = tmp_path_factory.mktemp("blocks") / "block_choice_host"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", str(cuda), "-o", str(out),
                    str(ROOT / "tests" / "block_choice_host.cpp")], check=True)
    return out


@pytest.mark.parametrize("ms,want", [
    ((1.0, 1.1, 1.2, 1.3), (0, 64)),        # by size is fastest
    ((1.0, 1.2, 1.0, 1.3), (0, 128)),       # a tie
    ((1.0, 1.2, 0.99, 1.3), (0, 128)),      # within what timings differ
    ((1.0, 1.2, 1.1, 0.9), (256, 256)),     # a fixed size is faster
    ((1.0, 0.9, 0.95, 0.0), (64, 64)),      # 256 is not tried for every kernel
    ((1.0, 1.1, 1.05, 0.0), (0, 128)),
    ((0.0, 0.0, 0.0, 0.0), (0, 64))])       # nothing launched (the rates of two or three species)
def test_choice(program, ms, want):
    r = subprocess.run([str(program), *map(str, ms)], capture_output=True, text=True, check=True)
    assert tuple(int(v) for v in r.stdout.split()) == want
