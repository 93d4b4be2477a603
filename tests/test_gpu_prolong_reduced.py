"""Warm start from an energy-band grid, and target nodes: every node of the destination accounted for.

The source's value is M-like outside its node set: a cell with a corner outside
gives the destination's penalty, and a nearest node outside the code 0.  Target
nodes come from the destination's own target box: exactly those are 0.  Sizes
below a block's round and past a whole round of the grid with a rest.
Reference: Q1 interpolation in numpy FP64, 1e-12 of the largest corner as in the
box tests; nodes whose foot is within 1e-9 of a node of the source (a face) or
halfway between two (the code) are decided by an ulp and left out there.
"""
import numpy as np
import pytest

from paper_2407_14675_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reduced", [0, 1])
@pytest.mark.parametrize("n_dst", [(10, 11, 12, 6), (22, 24, 19, 20)])
def test_every_node_of_the_destination(dp, n_dst, reduced):
    src = W.config2(n=17).replace(n=(17, 15, 16, 5), precision=W.FP64, reduced=reduced)
    dst = W.config1().replace(n=n_dst, precision=W.FP64, target_w=(0.03, 0.03, 0.03, 0.0))
    rng = np.random.default_rng(5)
    V = rng.uniform(0.5, 1.0, size=src.nodes)
    codes = W.random_codes(src, 4)
    codes[codes == 0] = 1
    with dp.Grid(src) as s, dp.Grid(dst) as d:
        idx = s.active_index()
        s.set_value(V[idx])
        s.set_policy(codes[idx])
        stored = s.get_value()
        dp.dp_warm_start_from_grid(s.h, d.h)
        got_v, got_c, M = d.get_value(), d.get_policy(), d.info["penalty_M"]
    active = np.zeros(src.nodes, bool)
    active[idx] = True
    assert active.all() != bool(reduced)
    V = np.full(src.nodes, np.nan)
    V[idx] = stored
    V, active = V.reshape(src.n), active.reshape(src.n)
    cell, frac, near, edge, half, target = [], [], [], [], [], []
    for k in range(4):
        h_s, h_d = ((p.hi[k] - p.lo[k]) / (p.n[k] - 1) for p in (src, dst))
        x = dst.lo[k] + np.arange(dst.n[k]) * h_d
        u = (x - src.lo[k]) / h_s
        c = np.clip(np.floor(u).astype(int), 0, src.n[k] - 2)
        cell.append(c)
        frac.append(u - c)
        near.append(np.clip(np.floor(u + 0.5).astype(int), 0, src.n[k] - 1))
        edge.append(np.abs(u - np.round(u)) < 1e-9)
        half.append(np.abs(u - np.floor(u) - 0.5) < 1e-9)
        w = dst.target_w[k]
        target.append(np.abs(x - dst.target_c[k]) < w if w > 0 else np.ones(dst.n[k], bool))

    def grid(a, op):
        a = [v.reshape([-1 if d == k else 1 for d in range(4)]) for k, v in enumerate(a)]
        return op(op(a[0], a[1]), op(a[2], a[3]))

    target, edge, half = grid(target, np.logical_and), grid(edge, np.logical_or), grid(half, np.logical_or)
    want, whole = np.zeros(dst.n), np.ones(dst.n, bool)
    for m in range(16):
        at = np.ix_(*[cell[k] + (m >> k & 1) for k in range(4)])
        w = [frac[k] if m >> k & 1 else 1.0 - frac[k] for k in range(4)]
        whole &= active[at]
        want += np.nan_to_num(V[at]) * np.einsum("i,j,k,l->ijkl", *w)
    want = np.where(whole, want, M)
    got_v, got_c = got_v.reshape(dst.n), got_c.reshape(dst.n)
    assert target.any() and (got_v[target] == 0.0).all() and (got_c[target] == 0).all()
    free = ~target
    # the source's own target nodes are 0, so a value may be: not below its corners
    ok = np.abs(got_v - want) <= 1e-12 * np.where(whole, 1.0, M)
    assert ok[free & ~edge].all()
    stored_near = active[np.ix_(*near)]
    want_c = np.where(stored_near, codes.reshape(src.n)[np.ix_(*near)], 0)
    assert (got_c == want_c)[free & ~half].all()
    assert (free & ~edge & ~half).mean() > 0.3
    if reduced:
        assert 0.02 < (whole & free).mean() < 0.98 and not stored_near.all()
