"""Variants that tables or block sizes choose, on a nine-species box of 65
nodes (not a multiple of any block) after three steps:

* binary diffusivities beyond a factor of 32 (floating sums and solves instead
  of fixed-point ones) in the mixed mode, against the oracle: 1e-5 of each
  set's largest population (three steps of a few ten float roundings of 6e-8);
* the same tables, and ln A beyond 512 (floating exponents of the rates), in
  one persistent launch against lbm_step: the bounds of rounding of
  test_gpu_persistent.py, 1e-12 in double and 1e-6 in the float units;
* ln A beyond 512 on a reaction that does not proceed, against the mechanism
  without it: the same bounds (the fast mixed mode's floating rates, with
  exponentials to 3e-7, 1e-6 as well: a step changes no population by more
  than its own size);
* 64 and 128 threads per block of the double collision, against the oracle:
  1e-12, as the default's."""
import copy

import numpy as np
import pytest

import oracle
import workload as w

pytestmark = pytest.mark.gpu

STEPS = 3


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2101_01702_gb300 import build
    build.build()
    from paper_2101_01702_gb300 import lbm as L
    return L


def _precision(L, mode):
    return {"fp64": L.LBM_FP64, "mixed": L.LBM_MIXED, "fast": L.LBM_MIXED_FAST}[mode]


def _box(tables):
    prob = w.sphere3d_problem(shape=(13, 5, 1), radius=2.0)
    X = prob.init.X + np.array([0, 0, 0.02, 2e-3, 2e-3, 4e-3, 1e-4, 1e-4, 0])[:, None]
    prob.init.X = X / X.sum(axis=0)
    if tables == "wide_D":                  # 1/D_ab over a factor of 40
        D = prob.species.D.copy()
        D[0, 3] = D[3, 0] = D[0, 3] * 40.0
        prob.species.D = D
    elif tables == "small_A":               # H2 -> 2 H, forward only, with A = e^-600
        me = copy.copy(prob.mech)
        row = np.zeros((1, 9), dtype=np.int32)
        f, r = row.copy(), row.copy()
        f[0, 0], r[0, 3] = 1, 2
        me.nu_f, me.nu_r = np.concatenate([me.nu_f, f]), np.concatenate([me.nu_r, r])
        me.log_A = np.append(me.log_A, -600.0)
        me.b, me.theta = np.append(me.b, 0.0), np.append(me.theta, 0.0)
        me.rtype = np.append(me.rtype, 0).astype(np.int32)
        me.reversible = np.append(me.reversible, 0).astype(np.int32)
        me.eff = np.concatenate([me.eff, np.ones((1, 9))])
        me.low = np.concatenate([me.low, np.zeros((1, 3))])
        prob.mech = me
    return prob


def _run(L, prob, mode, launch="kernels", blocks=None):
    s = L.Solver.from_problem(prob, precision=_precision(L, mode))
    if blocks:
        s.set_blocks(blocks)
    if launch == "kernels":
        s.step(STEPS)
    else:
        s.step_persistent(STEPS, tile_mult=1)
    assert s.sync() == L.LBM_OK
    out = s.populations()
    s.close()
    return out


def _within(got, ref, tol):
    for k in range(ref.shape[0]):
        assert np.abs(got[k] - ref[k]).max() <= tol * np.abs(ref[k]).max(), k


def _oracle(prob):
    o = oracle.Oracle.from_problem(prob)
    assert o.step(STEPS) == 0
    return o.get_pop().transpose(1, 2, 0)


@pytest.mark.parametrize("mode", ["mixed", "fast"])
def test_wide_diffusivities_against_the_oracle(lbm, mode):
    prob = _box("wide_D")
    _within(_run(lbm, prob, mode), _oracle(prob), 1e-5)


@pytest.mark.parametrize("mode", ["fp64", "mixed", "fast"])
@pytest.mark.parametrize("tables", ["wide_D", "small_A"])
def test_persistent_equals_plain_steps(lbm, tables, mode):
    prob = _box(tables)
    _within(_run(lbm, prob, mode, "persistent"), _run(lbm, prob, mode), 1e-12 if mode == "fp64" else 1e-6)


@pytest.mark.parametrize("mode", ["fp64", "mixed", "fast"])
def test_floating_exponents_of_the_rates(lbm, mode):
    _within(_run(lbm, _box("small_A"), mode), _run(lbm, _box("plain"), mode), 1e-12 if mode == "fp64" else 1e-6)


@pytest.mark.parametrize("threads", [64, 128])
@pytest.mark.parametrize("tables", ["plain", "wide_D"])
def test_collision_blocks_against_the_oracle(lbm, tables, threads):
    prob = _box(tables)
    _within(_run(lbm, prob, "fp64", blocks=[128, 64, 64, 64, 64, threads]), _oracle(prob), 1e-12)
