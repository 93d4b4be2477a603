"""Work items of a batch: no setting and no tuning makes it slower than it was.

Evaluation launches share the nodes out equally, whatever item_eval says (one
item per transfer would leave most blocks without work).  The tuning of the
improvement items starts from the size in use: 256 nodes keep twice as many
blocks of a small batch busy as the smallest candidate, 512, and have to stay.
"""
import numpy as np
import pytest

from paper_2407_14675_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _ms(b, dp, mode):
    b.sweep(mode)
    return min(b.sweep(mode)[1] for _ in range(7))


def test_evaluation_does_not_depend_on_its_items(dp):
    probs = W.batch_transfers(count=6, seed=3, sizes=(21,))
    with dp.Batch(probs) as b:
        b.sweep(dp.DP_SWEEP_IMPROVE_FULL)
        ms = _ms(b, dp, dp.DP_SWEEP_EVAL)
        V = [b.get_value(k) for k in range(6)]
        dp.dp_batch_set_items(b.h, 1 << 20, b.info()["item_improve"])
        assert b.info()["item_eval"] == 1 << 20
        coarse = _ms(b, dp, dp.DP_SWEEP_EVAL)
        b.sweep(dp.DP_SWEEP_IMPROVE_FULL)
        assert np.isfinite(b.get_value(0)).all() and all((v >= 0).all() for v in V)
    print("evaluation sweep %.4f ms, with one item a transfer %.4f ms" % (ms, coarse))
    assert coarse <= 1.3 * ms


def test_tuning_keeps_the_item_in_use_unless_another_is_faster(dp):
    probs = W.batch_transfers(count=2, seed=5, sizes=(13,))
    with dp.Batch(probs) as b:
        dp.dp_batch_set_items(b.h, 8192, 256)
        b.sweep(dp.DP_SWEEP_IMPROVE_FULL)
        fine = _ms(b, dp, dp.DP_SWEEP_IMPROVE_WALK)
        dp.dp_batch_set_items(b.h, 8192, 512)
        coarse = _ms(b, dp, dp.DP_SWEEP_IMPROVE_WALK)
        print("walk sweep %.4f ms at 256 nodes an item, %.4f at 512" % (fine, coarse))
        dp.dp_batch_set_items(b.h, 8192, 256)
        assert b.autotune() == (8192, 256)
        assert (b.get_value(0) == 0).all()
