"""Stored diagonal factors of the FP64 evaluation (DP_SWEEP_EVAL_DIAG on FP64 grids).

The first diagonal-solved sweep after an improvement stores 1 / (1 - beta w_jj)
per node and the later ones read it.  Against the sweep that recomputes feet
and factors from the policy codes (the policy set from the host): the two
share every operation but the running cost's contraction, an ulp of the value
(test_gpu_diag.py's bound, 1e-13 of max|V|, per sweep).
"""
import numpy as np
import pytest

from paper_2407_14675_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _problem(kind):
    if kind == "polar":
        return W.example1(n=(9, 7, 6, 8))
    p = W.config0().replace(n=(13, 11, 9, 7), refine=1, n_angles=32)
    if kind == "band":
        lo, hi = W.energy_band(1.0, 1.05, margin=0.05)
        p = p.replace(reduced=1, energy_lo=lo, energy_hi=hi)
    return p


@pytest.mark.parametrize("kind", ["box", "band", "polar"])
def test_stored_factors_give_the_recomputed_sweeps(dp, kind):
    p = _problem(kind)
    with dp.Grid(p) as g, dp.Grid(p) as h:
        V = W.smooth_value(p, 3)[g.active_index()]
        g.set_value(V)
        for step in range(3):                       # new feet each time: the factors are stored anew
            g.sweep(dp.DP_SWEEP_IMPROVE_FULL if step == 0 else dp.DP_SWEEP_IMPROVE_WALK)
            h.set_value(g.get_value())
            h.set_policy(g.get_policy())
            for k in range(3):
                rg, rh = g.sweep(dp.DP_SWEEP_EVAL_DIAG), h.sweep(dp.DP_SWEEP_EVAL_DIAG)
                a, b = g.get_value(), h.get_value()
                tol = 1e-13 * (k + 1) * np.abs(b).max()
                assert np.abs(a - b).max() <= tol
                assert abs(rg - rh) <= tol


@pytest.mark.parametrize("kind", ["box", "band"])
def test_a_sweep_after_a_solve_that_stopped_on_the_device(dp, kind):
    """The sweep that would have stored the factors returns at the passed stopping test."""
    p = _problem(kind)
    with dp.Grid(p) as g, dp.Grid(p) as h:
        g.policy_iterate(tol=1e-6, max_sweeps=200, n_eval=20, eval_solver=dp.DP_EVAL_DIAG)
        V = W.smooth_value(p, 5)[g.active_index()]
        for x in (g, h):
            x.set_value(V)
        h.set_policy(g.get_policy())
        for k in range(2):
            g.sweep(dp.DP_SWEEP_EVAL_DIAG)
            h.sweep(dp.DP_SWEEP_EVAL_DIAG)
            assert np.abs(g.get_value() - h.get_value()).max() <= 1e-13 * (k + 1) * p.M()
