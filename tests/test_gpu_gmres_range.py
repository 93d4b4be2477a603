"""GMRES on FP32 grids with values near the end of FP32's range.

With values of about 1e18 the sum of squares of a warp's share of the residuals
(2,800 entries of 61^4) leaves FP32's range although every product and every
sum of 128 of them is inside.  The call has to converge as it does for the same
problem at 2^-40 of the size, where every operation is the same but for the
exponent and the cost: the next evaluation sweep moves the value by no more than
the tolerance then, the one before having moved it by less (a contraction).
"""
import pytest

from paper_2407_14675_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [2.0 ** -40, 1.0])
def test_values_near_the_end_of_the_range(dp, scale):
    M = 1.3e18 * scale
    p = W.config1(n=61).replace(penalty_M=M)
    with dp.Grid(p) as g:
        g.set_value(W.random_value(p, 3) * 0.5)
        g.set_policy(W.random_codes(p, 4))
        rc, st = g.policy_evaluate(tol=1e-4 * M, max_sweeps=400, gmres_restart=20)
        assert rc == dp.DP_OK and st.converged
        assert g.sweep(dp.DP_SWEEP_EVAL) <= 1e-4 * M
