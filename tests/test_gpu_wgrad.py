"""Network gradients at the batches where the weight gradients' ring and the fused reductions can go wrong.

512 rows: two splits of four 64-row chunks (the ring refills once); 1,536 and
2,560: splits of 256 rows, counts that are no power of two; 16,896: 22 splits of
768 rows, 132 row tiles of the persistent kernels.  Same reference and bounds as
the sizes of test_gpu_mlp.py.
"""
import pytest

from test_gpu_mlp import test_gradients_match_bf16_reference as _gradients_match

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [512, 1536, 2560, 16896])
def test_gradients_at_ring_edges(dp, n):
    _gradients_match(dp, n)
