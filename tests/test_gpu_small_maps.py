"""Exact dW of maps of fewer than 64 pixels, against the oracle: every filter, stride and layout form of the small-map kernels."""
import pytest
import torch

from oracle import oracle
from paper_1908_05460_b200 import binding as B
from paper_1908_05460_b200 import inputs as I
from paper_1908_05460_b200.layers import ConvLayer
from helpers import GpuLayer, norm_err, oshape, to_f64, TOL_F32

pytestmark = pytest.mark.gpu

SHAPES = [
    ConvLayer("1x1 filter, 16 channels on 4x4", 59, 16, 4, 4, 16, 1, 1, 1, 0, dy_std=1.0),
    ConvLayer("1x1 filter, 40 channels on 2x8", 33, 40, 2, 8, 24, 1, 1, 1, 0),
    ConvLayer("1x3 filter, 32 channels on 4x8", 9, 32, 4, 8, 72, 1, 3, 1, 0),
]


@pytest.mark.parametrize("layout", [dict(), dict(x_layout=B.X_NCHW, dw_layout=B.DW_KCRS), dict(dy_layout=B.DY_NPQK)], ids=["paper", "nchw", "nhwc"])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("li", range(len(SHAPES)), ids=[l.name for l in SHAPES])
def test_matches_the_oracle(li, dtype, layout):
    layer = SHAPES[li]
    x, dy = I.make_layer_inputs(layer, dtype, 15, li)
    ref, dn = oracle.dw_exact(to_f64(x), to_f64(dy), oshape(layer), 0.5)
    assert norm_err(GpuLayer(layer, dtype, x, dy, alpha=0.5, **layout).exact(), ref, dn) <= TOL_F32
