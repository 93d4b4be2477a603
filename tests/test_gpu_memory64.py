"""Device memory of FP64 grids: what every grid holds, and what a diagonal-solved evaluation adds.

Two value buffers, the policy and the frozen feet (16 + 2 + 48 bytes a node) and
for the polar dynamics the running cost (8); the diagonal factors (8 bytes a
node) come with the first evaluation that uses them, and only once.  Tables and
scratch of fixed size are allowed 1 MB.
"""
import numpy as np
import pytest

from paper_2407_14675_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,per_node", [("orbit", 66), ("polar", 74)])
def test_the_diagonal_factors_come_with_their_first_use(dp, kind, per_node):
    p = W.config0().replace(n=(21, 21, 21, 21)) if kind == "orbit" else W.example1(n=(24, 20, 20, 20))
    with dp.Grid(p) as g:
        held = lambda: dp.dp_grid_get_info(g.h)["device_bytes"]
        assert per_node * p.nodes <= held() <= per_node * p.nodes + (1 << 20)
        g.policy_iterate(tol=0.0, max_sweeps=2, n_eval=3)
        before = held()
        g.policy_iterate(tol=0.0, max_sweeps=2, n_eval=3, eval_solver=dp.DP_EVAL_DIAG)
        assert held() == before + 8 * p.nodes
        g.policy_iterate(tol=0.0, max_sweeps=2, n_eval=3, eval_solver=dp.DP_EVAL_DIAG)
        g.sweep(dp.DP_SWEEP_EVAL_DIAG)
        assert held() == before + 8 * p.nodes
        assert np.isfinite(g.get_value()).all()
