"""Feedback and closed loop where no angle compares: a code of the table, no access outside it.

A penalty beyond FP32's range makes it infinity on an FP32 grid, and the
differences of a state whose feet all leave the box NaN.  The result has no
meaning there, but the call returns: the first angle, and finite states.
"""
import numpy as np
import pytest

from paper_2407_14675_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("angles", [3, 64])
@pytest.mark.parametrize("refine", [0, 1])
def test_states_without_a_comparable_angle(dp, angles, refine):
    p = W.config1(n=9).replace(penalty_M=1e39, n_angles=angles, refine=refine)
    lo, hi = np.array(p.lo), np.array(p.hi)
    x = np.tile(0.5 * (lo + hi), (40, 1))
    x[::2, 3] = lo[3]                 # the mass leaves the box: every foot is outside
    with dp.Grid(p) as g:
        g.set_value(W.smooth_value(W.config1(n=9), 3))
        alpha, _ = g.feedback(x, p.dt)
        _, xf = g.simulate(x, p.dt, p.dt, 3 * p.dt)
    assert (alpha[::2] == 0.0).all()
    assert ((alpha >= 0) & (alpha < 2 * np.pi)).all() and np.isfinite(xf).all()
