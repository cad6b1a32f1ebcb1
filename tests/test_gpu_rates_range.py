"""Production rates whose exponents are near the end of the double range: a
reactant with g/(R_U T) between -707 and -709.1, where e^g is no longer in the
range of the integer reduction and c e^g is a normal double.  The forward rate
does not depend on g (it multiplies the reactant's activity and divides the
rate coefficient), so the closed form is A c_R c_O.  (A g of +707 and more
makes the activity itself infinite at these concentrations.)  Tolerance
1e-11: three exponents of 710 in units of 2^-53 and the tables' own rounding,
a few 1e-13."""
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


@pytest.mark.parametrize("mode", ["fp64", "mixed"])
@pytest.mark.parametrize("g", [-709.0, -707.5])
def test_activities_near_the_end_of_the_range(lbm, mode, g):
    prob = w.config1_problem()
    sp, me = prob.species, prob.mech
    me.log_A, me.theta = np.array([0.5]), np.array([0.0])
    sp.h_form = sp.h_form.copy()
    sp.h_form[0] = g * (sp.r_lat / sp.W[0]) * sp.T0            # g of the first reactant at T0
    s = lbm.Solver(prob.lattice, sp, me, precision=lbm.LBM_FP64 if mode == "fp64" else lbm.LBM_MIXED)
    T = sp.T0 * np.array([1.0 - 1e-4, 1.0, 1.0 + 1e-4])
    rho = np.array([[200.0], [320.0], [34.0]]) * np.ones(3)
    got = s.chemistry_at(rho, T)["rho_dot"]
    s.close()
    q = np.exp(me.log_A[0]) * (rho[0] / sp.W[0]) * (rho[1] / sp.W[1])
    for a, sign in ((0, -1.0), (1, -1.0), (2, 1.0)):
        assert np.abs(got[a] / (sign * sp.W[a] * q) - 1.0).max() <= 1e-11
