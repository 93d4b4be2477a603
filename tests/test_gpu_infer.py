"""Inference in one kernel: the grid route (dp_warm_start) against the state route (dp_mlp_forward).

Both run the same layers; they differ in where the inputs come from (a table
of normalised coordinates per dimension, or the states) and where the outputs
go.  The coordinates agree to one FP32 rounding, which moves an output by at
most the isolated BF16 rounding flips test_gpu_mlp.py bounds at 2e-3 of the
output scale.  The sizes cover one row, a tile's edge, ragged and reduced
grids, FP64 storage and more tiles than resident blocks.
"""
import numpy as np
import pytest

from paper_2407_14675_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL_Y = 2e-3


def _net(dp, p, cap=4096, seed=5):
    net = dp.Mlp(p.lo, p.hi, batch_capacity=cap)
    dp.dp_mlp_set_params(net.h, dp.flatten_params(W.mlp_init_params(seed=seed)))
    return net


def _nodes(p, idx):
    i = np.stack(np.unravel_index(idx, p.n), 1)
    return np.array(p.lo) + i * ((np.array(p.hi) - np.array(p.lo)) / (np.array(p.n) - 1))


@pytest.mark.parametrize("n,precision,reduced", [((2, 3, 5, 4), W.FP32, 0), ((4, 4, 4, 2), W.FP32, 0), ((9, 8, 7, 11), W.FP64, 0),
                                                 ((25, 25, 25, 25), W.FP32, 1), ((41, 23, 31, 19), W.FP32, 0)])
def test_warm_start_equals_forward_at_the_nodes(dp, n, precision, reduced):
    p = W.config1().replace(n=n, precision=precision)
    if reduced:
        lo, hi = W.energy_band(1.0, 1.05)
        p = p.replace(reduced=1, energy_lo=lo, energy_hi=hi)
    with dp.Grid(p) as g, _net(dp, p) as net:
        dp.dp_warm_start(net.h, g.h)
        V, code = g.get_value(), g.get_policy()
        x = _nodes(p, g.active_index())
        y = dp.dp_mlp_forward(net.h, x).astype(np.float64)
    scale = np.abs(y).max()
    c, w = np.array(p.target_c), np.array(p.target_w)
    tgt = ((np.abs(x - c) < w) | (w <= 0)).all(1)
    assert (V[tgt] == 0).all()
    want = p.M() * np.clip(y[:, 0], 0.0, 1.0)
    assert np.abs(V - want)[~tgt].max() <= TOL_Y * scale * p.M()
    size = np.hypot(y[:, 1], y[:, 2])
    off = np.angle(np.exp(1j * (code * (2 * np.pi / 65536) - np.arctan2(y[:, 2], y[:, 1]))))
    assert (np.abs(off) * size).max() <= TOL_Y * scale * 2 + size.max() * np.pi / 65536


@pytest.mark.parametrize("count", [1, 127, 128, 129, 4097])
def test_forward_rows_do_not_depend_on_the_count(dp, count):
    p = W.config1()
    rng = np.random.default_rng(3)
    x = np.array(p.lo) + (np.array(p.hi) - np.array(p.lo)) * rng.uniform(size=(5000, 4))
    with _net(dp, p, cap=8192) as net:
        whole = dp.dp_mlp_forward(net.h, x)
        assert (dp.dp_mlp_forward(net.h, x[:count]) == whole[:count]).all()
