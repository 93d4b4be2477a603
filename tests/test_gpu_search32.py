"""FP32 angle searches against the oracle's, over the tables and boxes where their bookkeeping can go wrong.

Tables whose brackets differ in length (K does not divide 65536), the smallest
table, the largest (its bracket is the shortest), ragged and tiny boxes whose
feet leave the cell and the box, and the reduced grid, whose cells may have a
corner outside (the penalty then sits in the corners).  The bounds are the
suite's: values within 1e-4 of max|V|, codes equal or a tie within 1e-5 M.
The evaluation at the feet that the search stored must equal the one at feet
formed anew from the codes.
"""
import numpy as np
import pytest

import oracle
from paper_2407_14675_gb300 import workloads as W
from test_gpu_parity import TOL32, _check_codes, _check_values

pytestmark = pytest.mark.gpu

CASES = [(dict(n=(9, 8, 7, 5)), 64), (dict(n=(6, 11, 5, 4)), 72), (dict(n=(7, 7, 9, 3)), 29), (dict(n=(5, 6, 9, 2)), 2),
         (dict(n=(8, 5, 6, 3), accel=5e-3), 1024), (dict(n=(13, 12, 11, 6), band=True), 48)]


@pytest.mark.parametrize("kw,angles", CASES)
@pytest.mark.parametrize("refine", [0, 1])
@pytest.mark.parametrize("walk", [False, True])
def test_fp32_search_parity(dp, kw, angles, refine, walk):
    kw = dict(kw)
    band = kw.pop("band", False)
    p = W.config1().replace(n_angles=angles, refine=refine, **kw)
    if band:
        e_lo, e_hi = W.energy_band(1.0, 1.05)
        p = p.replace(reduced=1, energy_lo=e_lo, energy_hi=e_hi)
    o = oracle.Oracle(p)
    V = W.smooth_value(p, 31).astype(np.float32).astype(np.float64)
    start = W.random_codes(p, 5)
    with dp.Grid(p) as g:
        idx = g.active_index()
        g.set_value(V[idx])
        g.set_policy(start[idx])
        g.sweep(dp.DP_SWEEP_IMPROVE_WALK if walk else dp.DP_SWEEP_IMPROVE_FULL)
        v_gpu, c_gpu = g.get_value(), g.get_policy()
        g.sweep(dp.DP_SWEEP_EVAL)
        v_feet = g.get_value()
    with dp.Grid(p) as g:
        g.set_value(v_gpu)
        g.set_policy(c_gpu)
        g.sweep(dp.DP_SWEEP_EVAL)
        v_codes = g.get_value()
    Vo = V.copy()
    Vo[o.target.astype(bool)] = 0
    Vf = np.full(o.N, o.M)
    Vf[idx] = Vo[idx]
    W1, c_or, _, _ = o.sweep(Vf, mode=oracle.IMPROVE_WALK if walk else oracle.IMPROVE_FULL, codes=start if walk else None)
    live = ~o.target.astype(bool)[idx]
    _check_codes(o, Vf, idx[live], c_gpu[live], c_or[idx][live], tie=1e-5 * o.M)
    _check_values(v_gpu, W1[idx], TOL32, "search fp32")
    # the stored feet hold 18-bit fractions: V changes by at most max|V| over three of them
    assert np.abs(v_feet - v_codes).max() <= 3 * 2.0 ** -18 * np.abs(v_gpu).max()
