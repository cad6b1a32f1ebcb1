"""Steps with two or three species launch four kernels: the diffusion
velocities follow the moments in one, the production rates precede the energy
collision in another (their agreement with the oracle: test_gpu_parity.py).
Every block size gives the same bits on a lattice of 257 nodes (a block of one
node after full ones), and the time between the events around the production
rates is that of no launch, as for the ghost nodes of a periodic lattice (2 us;
10 to 12 with a kernel)."""
import numpy as np
import pytest

import workload as w

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2101_01702_gb300 import build
    build.build()
    from paper_2101_01702_gb300 import lbm as L
    return L


def _solver(L, mode, **kw):
    return L.Solver.from_problem(w.config1_problem(**kw), precision={
        "fp64": L.LBM_FP64, "mixed": L.LBM_MIXED, "fast": L.LBM_MIXED_FAST}[mode])


@pytest.mark.parametrize("mode", ["fp64", "mixed", "fast"])
def test_no_launch_for_the_rates(lbm, mode):
    s = _solver(lbm, mode)
    s.step(10)
    ph = s.step_timed(200)
    s.close()
    assert ph[2] <= 2.0 * ph[0]


@pytest.mark.parametrize("mode", ["fp64", "mixed", "fast"])
def test_blocks_do_not_matter(lbm, mode):
    out = []
    for blocks in (None, [128, 64, 64, 64, 64, 64], [128, 128, 256, 128, 128, 128], [128, 128, 64, 256, 256, 64]):
        s = _solver(lbm, mode, nx=257, ny=1, nz=1)
        if blocks:
            s.set_blocks(blocks)
        s.step(3)
        out.append(s.populations())
        s.close()
    assert np.isfinite(out[0]).all()
    for o in out[1:]:
        np.testing.assert_array_equal(o, out[0])
