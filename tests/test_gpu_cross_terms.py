"""Cross terms of the double collision (sum over partner species of the
quasi-equilibrium differences): the fixed-point sums, used while the binary
diffusivities lie within a factor of 32, the floating sums beyond it, and
three species (floating sums always), each against the oracle after three
steps, on a box with 33, 64 and 65 nodes in turn so that the last block of
64 threads is empty, full and partly filled.  Tolerance: 1e-12 of each
set's largest population, the bound of the periodic parity tests (three
steps of a few hundred roundings of 1.1e-16 each).  A species that is
absent (exactly zero) is created by the reactions as one present at 1e-40
is."""
import numpy as np
import pytest

import oracle
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


def _box(shape, spread):
    prob = w.sphere3d_problem(shape=shape, radius=2.0)
    X = prob.init.X + np.array([0, 0, 0.02, 2e-3, 2e-3, 4e-3, 1e-4, 1e-4, 0])[:, None]
    prob.init.X = X / X.sum(axis=0)
    if spread != 1.0:                       # 1/D_ab over a wider range, symmetric
        D = prob.species.D.copy()
        D[0, 3] = D[3, 0] = D[0, 3] * spread
        prob.species.D = D
    return prob


@pytest.mark.parametrize("shape", [(11, 3, 1), (4, 4, 4), (13, 5, 1)])
@pytest.mark.parametrize("spread", [1.0, 6.0, 40.0])
def test_nine_species_against_the_oracle(lbm, shape, spread):
    prob = _box(shape, spread)
    o = oracle.Oracle.from_problem(prob)
    assert o.step(3) == 0
    ref = o.get_pop().transpose(1, 2, 0)
    s = lbm.Solver.from_problem(prob, precision=lbm.LBM_FP64)
    s.step(3)
    got = s.populations()
    s.close()
    for k in range(ref.shape[0]):
        assert np.abs(got[k] - ref[k]).max() <= 1e-12 * np.abs(ref[k]).max(), k


def test_three_species_against_the_oracle(lbm):
    prob = w.config1_problem(nx=13, ny=5, nz=1, slab=(5, 8))
    o = oracle.Oracle.from_problem(prob)
    assert o.step(3) == 0
    ref = o.get_pop().transpose(1, 2, 0)
    s = lbm.Solver.from_problem(prob, precision=lbm.LBM_FP64)
    s.step(3)
    got = s.populations()
    s.close()
    for k in range(ref.shape[0]):
        assert np.abs(got[k] - ref[k]).max() <= 1e-12 * np.abs(ref[k]).max(), k


def test_absent_species_keeps_its_source(lbm):
    prob = _box((4, 4, 4), 1.0)
    got = []
    for x in (0.0, 1e-40):
        prob.init.X[3] = x                  # H
        s = lbm.Solver.from_problem(prob, precision=lbm.LBM_FP64)
        s.step(1)
        got.append(s.populations())
        s.close()
    assert np.abs(got[1][3]).max() > 0
    for k in range(got[0].shape[0]):
        assert np.abs(got[0][k] - got[1][k]).max() <= 1e-12 * np.abs(got[1][k]).max(), k
