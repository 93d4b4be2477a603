"""Warm start of a grid from another grid's value: the tabulated cells, fractions and nearest nodes.

The largest dimension (1,024 nodes) on either side, grids smaller than a block
and larger than a round of blocks, a destination that reaches outside the
source's box, and the periodic angle.  Reference: the same Q1 interpolation in
numpy FP64, value within 1e-12 of its largest corner (15 lerps at 2^-53 each),
nearest node and outside test exact.
"""
import numpy as np
import pytest

from paper_2407_14675_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [((1024, 2, 2, 3), (2, 3, 2, 1024), 0.0, False), ((3, 2, 1024, 2), (1024, 3, 3, 2), 0.05, False),
         ((2, 3, 2, 2), (5, 3, 4, 2), 0.0, False), ((9, 8, 7, 5), (31, 29, 27, 25), 0.02, False),
         ((7, 6, 5, 8), (13, 11, 9, 15), 0.0, True)]


@pytest.mark.parametrize("n_src,n_dst,grow,polar", CASES)
def test_values_and_codes_of_the_destination(dp, n_src, n_dst, grow, polar):
    if polar:
        src, dst = W.example1(n=n_src), W.example1(n=n_dst)
    else:
        src = W.config1().replace(n=n_src, precision=W.FP64)
        lo, hi = np.array(src.lo), np.array(src.hi)
        dst = src.replace(n=n_dst, lo=tuple(lo - grow * (hi - lo)), hi=tuple(hi + grow * (hi - lo)))
    V = np.random.default_rng(2).uniform(0.0, 1.0, size=src.nodes)
    codes = W.random_codes(src, 4)
    with dp.Grid(src) as s, dp.Grid(dst) as d:
        s.set_value(V)
        s.set_policy(codes)
        V = s.get_value()     # target nodes are 0
        dp.dp_warm_start_from_grid(s.h, d.h)
        got_v, got_c, M = d.get_value(), d.get_policy(), d.info["penalty_M"]
    cell, frac, near, out, face, tie = [], [], [], [], [], []
    for k in range(4):
        def spacing(p):
            return (p.hi[k] - p.lo[k]) / (p.n[k] - 1)
        x = dst.lo[k] + np.arange(dst.n[k]) * spacing(dst)
        u = (x - src.lo[k]) / spacing(src)
        f = np.floor(u)
        c, t = f.astype(int), u - f
        if polar and k == 3:
            o = np.zeros(len(u), bool)
            c %= src.n[k]
            q = np.floor(u + 0.5).astype(int) % src.n[k]
        else:
            o = (u < 0) | (u > src.n[k] - 1)
            top = (c > src.n[k] - 2) | (c < 0)
            c, t = np.where(top, src.n[k] - 2, c), np.where(top, 1.0, t)
            q = np.clip(np.floor(u + 0.5).astype(int), 0, src.n[k] - 1)
        cell.append(c)
        frac.append(t)
        near.append(q)
        out.append(o)
        # an ulp decides on the box's face, and halfway between two nodes
        face.append((np.abs(u) < 1e-9) | (np.abs(u - (src.n[k] - 1)) < 1e-9))
        tie.append(np.abs(u - np.floor(u) - 0.5) < 1e-9)
    V4 = V.reshape(src.n)
    want = np.zeros(dst.n)
    for m in range(16):
        idx = [(cell[k] + (m >> k & 1)) % src.n[k] for k in range(4)]
        w = [frac[k] if m >> k & 1 else 1.0 - frac[k] for k in range(4)]
        want += V4[np.ix_(*idx)] * np.einsum("i,j,k,l->ijkl", *w)

    def anywhere(a):
        return (a[0][:, None, None, None] | a[1][None, :, None, None] | a[2][None, None, :, None] | a[3]).reshape(-1)

    inside = want.reshape(-1)
    want = np.where(anywhere(out), M, inside)
    target = got_v == 0.0
    err = np.abs(got_v - want)
    either = np.minimum(err, np.abs(got_v - np.where(anywhere(out), inside, M)))
    err = np.where(anywhere(face), either, err)
    assert err[~target].max() <= 1e-12 * max(1.0, M)
    assert (got_c == codes.reshape(src.n)[np.ix_(*near)].reshape(-1))[~target & ~anywhere(tie)].all()
    assert target.mean() < 0.9
