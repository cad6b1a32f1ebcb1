"""Species that start at exactly zero: the reactions create them at levels
below the smallest normal float, and a front of such densities crosses the
lattice.  The steps of the mixed modes stay finite, report no error and keep
the bound of the mixed modes (1e-4 of each field's largest value) against the
double step, in kernels of their own and in one persistent launch."""
import numpy as np
import pytest

import workload as w

pytestmark = pytest.mark.gpu

STEPS = 30


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2101_01702_gb300 import build
    build.build()
    from paper_2101_01702_gb300 import lbm as L
    return L


@pytest.fixture(scope="module")
def problem():
    prob = w.sphere3d_problem(shape=(64, 5, 4), radius=3.0)
    X = prob.init.X.copy()
    X[2:8] = 0.0                                   # all but H2, O2 and N2
    prob.init.X = X / X.sum(axis=0)
    return prob


@pytest.fixture(scope="module")
def reference(lbm, problem):
    s = lbm.Solver.from_problem(problem, precision=lbm.LBM_FP64)
    s.step(2)
    early = s.moments(lbm.LBM_F_RHO_A)["rho_a"]
    # the state the test is about: nodes on either side of the smallest normal and subnormal floats
    tiny = (np.abs(early[2:8]) < 1.2e-38) & (early[2:8] != 0)
    assert tiny.sum() > 100
    s.step(STEPS - 2)
    m = s.moments(lbm.LBM_F_T | lbm.LBM_F_Y)
    s.close()
    return m


@pytest.mark.parametrize("launch", ["kernels", "persistent"])
@pytest.mark.parametrize("mode", ["mixed", "mixed_fast"])
def test_species_from_zero(lbm, problem, reference, mode, launch):
    s = lbm.Solver.from_problem(problem, precision=lbm.LBM_MIXED if mode == "mixed" else lbm.LBM_MIXED_FAST)
    if launch == "kernels":
        s.step(STEPS)
    else:
        s.step_persistent(STEPS)
    assert s.sync() == lbm.LBM_OK
    m = s.moments(lbm.LBM_F_T | lbm.LBM_F_Y)
    assert np.isfinite(s.populations()).all()
    s.close()
    for k in ("T", "Y"):
        top = np.abs(reference[k]).max(axis=-1, keepdims=True)
        assert (np.abs(m[k] - reference[k]) <= 1e-4 * top).all(), (k, (np.abs(m[k] - reference[k]) / top).max())
