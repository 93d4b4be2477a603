"""FP64 angle searches decided by the FP32 model against the search that evaluates every angle.

The value after a sweep must be the oracle's (FP64, every angle evaluated) to
1e-12 of M, the suite's bound for a tie of two controls, so a wrong decision
shows wherever it costs anything.  The fields stress the model: smooth, rough
(every cell its own slopes), flat (all ties) and flat with jumps; the boxes are
ragged and tiny, so that feet leave them; tables have from 2 to 72 angles
(below 30 the refinement does not use the model), and the thrust ranges from
none to one that carries the foot across half a cell.  Where equal values make
the path of a walk or the bracket of a refinement arbitrary (the field with
jumps) only the tabulations are compared.
"""
import numpy as np
import pytest

import oracle
from paper_2407_14675_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _field(p, what):
    if what == "smooth":
        return W.smooth_value(p, 7)
    if what == "rough":
        return W.random_value(p, 8)
    if what == "flat":
        return np.full(p.nodes, 0.25 * p.M())
    return np.round(W.smooth_value(p, 9) / p.M() * 3) * p.M() / 3


CASES = [((9, 8, 7, 5), 64, 1e-3), ((6, 11, 5, 4), 72, 2e-2), ((7, 7, 7, 3), 30, 0.3), ((5, 6, 9, 4), 29, 1e-3),
         ((2, 3, 4, 2), 16, 1e-2), ((8, 5, 6, 3), 2, 1e-3), ((7, 6, 5, 4), 48, 0.0)]


@pytest.mark.parametrize("what", ["smooth", "rough", "flat", "steps"])
@pytest.mark.parametrize("n,angles,accel", CASES)
@pytest.mark.parametrize("refine", [0, 1])
def test_codes_and_values_of_the_searches(dp, n, angles, accel, refine, what):
    p = W.config0().replace(n=n, n_angles=angles, accel=accel, refine=refine)
    o = oracle.Oracle(p)
    V = _field(p, what)
    V[o.target.astype(bool)] = 0.0
    start = W.random_codes(p, 4)
    modes = [(dp.DP_SWEEP_VI, oracle.VI)]
    if what != "steps" or not refine:
        modes.append((dp.DP_SWEEP_IMPROVE_FULL, oracle.IMPROVE_FULL))
    if what != "steps":
        modes.append((dp.DP_SWEEP_IMPROVE_WALK, oracle.IMPROVE_WALK))
    with dp.Grid(p) as g:
        for mode, omode in modes:
            g.set_value(V)
            g.set_policy(start)
            g.sweep(mode)
            want = o.sweep(V, omode, None if omode == oracle.VI else start)[0]
            assert np.abs(g.get_value() - want).max() <= 1e-12 * p.M()
