"""Top-k selection around the sizes where it changes how it holds a map, and the tiled transposition in front of the
gather at the edges of its tiles."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_1908_05460_b200 import binding as B
from paper_1908_05460_b200 import inputs as I
from paper_1908_05460_b200.layers import ConvLayer
from helpers import GpuLayer, to_f64

pytestmark = pytest.mark.gpu
DTYPES = pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])


@DTYPES
@pytest.mark.parametrize("pq", [(1, 1), (1, 32), (3, 11), (8, 8), (5, 13), (11, 12), (16, 16), (17, 16), (24, 32), (7, 110), (32, 32), (25, 41)])
def test_selection_with_ties(dtype, pq):
    layer = ConvLayer("select", 3, 4, pq[0], pq[1], 11, 1, 1, 1, 0)
    x, dy = I.make_layer_inputs(layer, dtype, 13, 0)
    dy = torch.round(dy.float() / dy.float().std() * 2).to(dtype)         # few distinct magnitudes, both signs, zeros
    topk = min(8, pq[0] * pq[1])
    idx, s = GpuLayer(layer, dtype, x, dy, topk=topk).select_topk()
    idx_ref, sum_ref, _ = oracle.topk_select(to_f64(dy), topk)
    np.testing.assert_array_equal(idx, idx_ref)
    np.testing.assert_array_equal(s, sum_ref)                              # small whole numbers: every order gives the same sum


@DTYPES
@pytest.mark.parametrize("c,hw", [(8, (5, 13)), (64, (8, 8)), (72, (16, 17)), (136, (7, 9)), (4, (12, 16)), (60, (1, 3))])
def test_transposed_activations(dtype, c, hw):
    layer = ConvLayer("transposed", 5, c, hw[0], hw[1], 16, 3, 3, 1, 1)
    x, dy = I.make_layer_inputs(layer, dtype, 14, 0)
    np.testing.assert_array_equal(GpuLayer(layer, dtype, x, dy, x_layout=B.X_NCHW).approx(B.METHOD_TOP1), GpuLayer(layer, dtype, x, dy).approx(B.METHOD_TOP1))
