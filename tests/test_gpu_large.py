"""An FP64 grid of more than 2^30 nodes: every sweep reaches all of it and nothing else.

1,107,296,256 nodes (73 GB).  The FP64 searches launch a thread a node, so a node
and the launch's stride add up to more than 2^31.  From V = 0 the value after k
sweeps is dt (1 + beta + ... + beta^(k-1)) wherever the feet of k steps stay in
the box and off the target, which the feedback's value at states all over the
box shows: tau + beta I[V] there.  Bound: k roundings of 2^-53 and the blend's.
"""
import numpy as np
import pytest

from paper_2407_14675_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_sweeps_cover_more_than_2_30_nodes(dp):
    p = W.config0().replace(n=(1024, 1024, 32, 33), target_c=(0.9, 0.0, 0.0, 0.0))
    assert p.nodes > 2 ** 30
    rng = np.random.default_rng(1)
    lo, hi = np.array(p.lo), np.array(p.hi)
    x = lo + (hi - lo) * np.stack([np.linspace(0.1, 0.9, 400), np.full(400, 0.5), np.full(400, 0.5),
                                   rng.uniform(0.3, 0.9, 400)], axis=1)
    x[:, 2] = x[:, 0] ** -0.5                        # circular orbits: the feet stay near
    with dp.Grid(p) as g:
        want = 0.0
        for k, mode in enumerate((dp.DP_SWEEP_VI, dp.DP_SWEEP_IMPROVE_WALK, dp.DP_SWEEP_EVAL, dp.DP_SWEEP_EVAL_DIAG)):
            g.sweep(mode)
            if mode != dp.DP_SWEEP_EVAL_DIAG:
                want = p.dt + p.beta * want
                _, q = g.feedback(x, p.dt)
                assert np.abs(q - (p.dt + p.beta * want)).max() <= 1e-14, k
            else:
                # a node's own coefficient solved: not below the plain update, not above the fixed point
                _, q = g.feedback(x, p.dt)
                assert ((q >= p.dt + p.beta * want - 1e-14) & (q <= p.dt / (1.0 - p.beta))).all()
