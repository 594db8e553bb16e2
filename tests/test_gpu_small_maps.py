"""Exact dW of maps of fewer than 64 pixels and of the smallest layers, against the oracle: every filter, stride and layout form of their kernels."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_1908_05460_b200 import binding as B
from paper_1908_05460_b200 import inputs as I
from paper_1908_05460_b200.layers import ConvLayer
from helpers import GpuLayer, kernel_names, norm_err, oshape, to_f64, TOL_F32

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


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("layer", [
    ConvLayer("1x1, three channels, rows of 36", 5, 3, 36, 36, 80, 1, 1, 1, 0),
    ConvLayer("1x1, rows of 64, one row a band", 2, 3, 3, 64, 17, 1, 1, 1, 0),
    ConvLayer("1x1, rows of 65, in two", 2, 2, 5, 65, 20, 1, 1, 1, 0),
    ConvLayer("1x1, whole maps of 25", 9, 4, 5, 5, 33, 1, 1, 1, 0),
    ConvLayer("3x3, rows of 38, unequal bands", 3, 3, 33, 38, 16, 3, 3, 1, 1),
    ConvLayer("3x3, stride 2, no padding", 3, 3, 31, 67, 19, 3, 3, 2, 0),
    ConvLayer("5x5 on one pixel", 7, 1, 5, 5, 3, 5, 5, 1, 0),
    ConvLayer("20 channels, odd rows", 2, 20, 9, 11, 20, 3, 3, 1, 1),
], ids=lambda l: l.name)
def test_small_layers_on_the_fp32_pipes(layer, dtype):
    """Bands and windows that are filled element by element: their edges, remainders of eight loads a thread, every memory order."""
    x, dy = I.make_layer_inputs(layer, dtype, 24, 0)
    ref, dn = oracle.dw_exact(to_f64(x), to_f64(dy), oshape(layer), 0.5)
    for kw in ({}, dict(x_layout=B.X_NCHW, dw_layout=B.DW_KCRS), dict(algo=B.ALGO_DIRECT)):
        g = GpuLayer(layer, dtype, x, dy, alpha=0.5, **kw)
        got = g.exact()
        assert norm_err(got, ref, dn) <= TOL_F32, kw
        np.testing.assert_array_equal(got, g.exact())
    assert any("direct_tiled_kernel" in n for n in kernel_names(lambda: B.gaconv_dw_exact(g.x, g.dy, g.dw, g.desc)))
