"""States that arrive early take no decisions after that.

On an FP64 grid a decision occupies the FP64 pipe of its SM.  Eight states share
a block in a call of eight per SM; seven of each eight start in the target and
arrive in the first step, the eighth flies on.  The call has to take about as
long as the late flights on their own (one warp's decision a step): an eighth
of the decisions is left, and a factor of 1.6 allows for the larger blocks.
The results are those of the late flights on their own.
"""
import time

import numpy as np
import pytest

from paper_2407_14675_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _best(f, times=5):
    f()
    t = []
    for _ in range(times):
        t0 = time.perf_counter()
        out = f()
        t.append(time.perf_counter() - t0)
    return min(t), out


def test_arrived_states_leave_the_pipe_to_the_others(dp):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    p = W.config0().replace(n_angles=64, refine=1)
    late = np.tile(np.array([0.96, 0.0, 0.96 ** -0.5, 0.99]), (sms, 1))
    late[:, 0] += np.linspace(0.0, 0.02, sms)
    x = np.tile(np.array([p.target_c[0], p.target_c[1], p.target_c[2], 0.99]), (8 * sms, 1))
    x[::8] = late
    with dp.Grid(p) as g:
        g.policy_iterate(tol=0.0, max_sweeps=2, n_eval=10)
        steps = 200
        alone, (t_one, x_one) = _best(lambda: g.simulate(late, p.dt, p.dt, steps * p.dt))
        mixed, (t_all, x_all) = _best(lambda: g.simulate(x, p.dt, p.dt, steps * p.dt))
    assert (t_all[::8] == -1.0).all()
    early = np.arange(8 * sms) % 8 != 0
    assert (t_all[early] == p.dt).all()
    np.testing.assert_array_equal(t_all[::8], t_one)
    np.testing.assert_array_equal(x_all[::8], x_one)
    print("late flights alone %.3f ms, with the early ones %.3f ms" % (1e3 * alone, 1e3 * mixed))
    assert mixed <= 1.6 * alone
