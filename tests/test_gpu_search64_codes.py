"""Codes of the FP64 searches against the oracle: long displacements, the reduced band and rough polar fields.

A dimension of 1,024 nodes takes the foot up to 400 cells (radial velocity)
and 100 (the periodic angle), past the reach of a frozen foot's 8-bit offsets;
the band has cells with corners outside the node set.  As in the parity tests,
a code counts as the oracle's when it is equal or ties it to 1e-12 of M by the
oracle's own value at both, at 99.9 % of the nodes; where a tie turned a
refinement to another bracket (the rest) the values still agree to 1e-6 of M.
"""
import numpy as np
import pytest

import oracle
from paper_2407_14675_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _problem(what):
    if what == "long v_r":
        return W.config0().replace(n=(6, 1024, 5, 4), dt=0.4, accel=2e-6, n_angles=64, refine=1)
    if what == "long theta":
        p = W.example1(n=(6, 5, 5, 1024))
        return p.replace(lo=(6800.0, -0.3, 7.4, 0.0), hi=(7200.0, 0.3, 7.7, p.hi[3]), dt=600.0)
    if what == "band":
        return W.config2(n=21).replace(precision=W.FP64)
    return W.example1(n=(20, 7, 7, 8))


@pytest.mark.parametrize("field", ["smooth", "rough"])
@pytest.mark.parametrize("what", ["long v_r", "long theta", "band", "polar"])
def test_codes_are_the_oracles(dp, what, field):
    p = _problem(what)
    o = oracle.Oracle(p)
    start = W.random_codes(p, 4)
    with dp.Grid(p) as g:
        idx = g.active_index()
        V = np.full(o.N, o.M)
        V[idx] = (W.smooth_value(p, 7) if field == "smooth" else W.random_value(p, 8))[idx]
        V[o.target.astype(bool)] = 0.0
        free = idx[~o.target[idx].astype(bool)]
        at = np.flatnonzero(~o.target[idx].astype(bool))
        for mode, omode in ((dp.DP_SWEEP_IMPROVE_FULL, oracle.IMPROVE_FULL),
                            (dp.DP_SWEEP_IMPROVE_WALK, oracle.IMPROVE_WALK)):
            g.set_value(V[idx])
            g.set_policy(start[idx])
            g.sweep(mode)
            want_v, want_c = o.sweep(V, omode, start)[:2]
            got_c = g.get_policy()[at]
            gap = np.abs(o.q_nodes(V, free, got_c) - o.q_nodes(V, free, want_c[free]))
            err = np.abs(g.get_value()[at] - want_v[free])
            assert ((got_c == want_c[free]) | (gap <= 1e-12 * o.M)).mean() >= 0.999
            assert (err <= 1e-12 * o.M).mean() >= 0.999 and err.max() <= 1e-6 * o.M
