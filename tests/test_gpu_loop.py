"""Closed loops whose states share a block's FP64 work against flying each state on its own.

A call with one state gives it a block; larger calls give a block two, four or
eight states, whose first warp does the FP64 work of all of them.  The counts
lie at and around the sizes where a block holds more, with states that arrive
early, late and never, and the results must be the same bits.
"""
import numpy as np
import pytest

from paper_2407_14675_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["box", "band", "fp64", "polar"])
@pytest.mark.parametrize("count", [2, 153, 305, 609, 1221])
def test_trajectories_do_not_depend_on_their_company(dp, what, count):
    p = {"box": W.config1(n=13), "band": W.config2(n=21), "fp64": W.config0().replace(n=(9, 9, 9, 9)),
         "polar": W.example1(n=(20, 7, 7, 8))}[what]
    lo, hi = np.array(p.lo), np.array(p.hi)
    x = lo + (hi - lo) * np.random.default_rng(count).uniform(0.2, 0.8, size=(count, 4))
    if what != "polar":
        # a third start beside the target
        t = np.array([p.target_c[d] if p.target_w[d] > 0 else x[0, d] for d in range(4)])
        x[::3] = t + (x[::3] - t) * 0.05
    with dp.Grid(p) as g:
        g.policy_iterate(tol=0.0, max_sweeps=2, n_eval=10, polish=0)
        t_all, x_all = g.simulate(x, p.dt, p.dt, 12 * p.dt)
        a_all, q_all = g.feedback(x, p.dt)
        for k in sorted({0, 1, count // 2, count - 2, count - 1} | set(range(0, count, max(1, count // 16)))):
            t_one, x_one = g.simulate(x[k:k + 1], p.dt, p.dt, 12 * p.dt)
            a_one, q_one = g.feedback(x[k:k + 1], p.dt)
            assert t_one[0] == t_all[k]
            np.testing.assert_array_equal(x_one[0], x_all[k])
            np.testing.assert_array_equal(a_one[0], a_all[k])
            assert q_one[0] == q_all[k]
