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
    """Bands and windows that are filled element by element: their edges, remainders of four loads a thread, every memory order."""
    x, dy = I.make_layer_inputs(layer, dtype, 24, 0)
    ref, dn = oracle.dw_exact(to_f64(x), to_f64(dy), oshape(layer), 0.5)
    orders = ({}, dict(x_layout=B.X_NCHW, dw_layout=B.DW_KCRS), dict(dy_layout=B.DY_NPQK), dict(x_layout=B.X_NCHW, dy_layout=B.DY_NPQK, dw_layout=B.DW_RSCK))
    for kw in (*orders, *(dict(o, algo=B.ALGO_DIRECT) for o in orders)):
        g = GpuLayer(layer, dtype, x, dy, alpha=0.5, **kw)
        got = g.exact()
        assert norm_err(got, ref, dn) <= TOL_F32, kw
        np.testing.assert_array_equal(got, g.exact())
        if "algo" in kw:
            assert any("direct_tiled_kernel" in n for n in kernel_names(lambda: B.gaconv_dw_exact(g.x, g.dy, g.dw, g.desc))), kw


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("x_layout,w", [(B.X_NHWC, 800_000), (B.X_NCHW, 2_400_000)], ids=["nhwc", "nchw"])
@pytest.mark.parametrize("rows", [1920, 640], ids=["64-bit offsets", "32-bit offsets"])
def test_windows_that_reach_far(rows, x_layout, w, dtype):
    """One wide row of X in the middle of `rows` rows of padding, one column of outputs: the offset of its pixel within a window, 944 or 304 rows
    of 2.4 million elements, takes more than 31 bits, or less."""
    n, c, k = 2, 3, 5
    gen = torch.Generator().manual_seed(28)
    x, dy = torch.randn((n, c), generator=gen).to(dtype), torch.randn((n, k, 2 * rows // 16 + 1), generator=gen).to(dtype)
    d = B.make_desc(ConvLayer("one row", n, c, 1, w, k, 1, 1, 1, 0), dtype, x_layout=x_layout, algo=B.ALGO_DIRECT)
    d.stride_h, d.stride_w, d.pad_h = 16, w, rows                     # (one column; the pixel is the middle output's)
    xg = torch.full((n, 1, w, c) if x_layout == B.X_NHWC else (n, c, 1, w), float("nan"), dtype=dtype, device="cuda")
    (xg[:, 0, 0, :] if x_layout == B.X_NHWC else xg[:, :, 0, 0]).copy_(x)
    dw, ws = torch.full((k, c), float("nan"), device="cuda"), B.attach_workspace(d, methods=(B.METHOD_EXACT,))
    B.gaconv_dw_exact(xg, dy.cuda(), dw, d)
    want = torch.einsum("nk,nc->kc", dy[:, :, rows // 16].double(), x.double())
    assert float((dw.cpu().double() - want).abs().max()) <= 1e-5 and B.gaconv_poll_async_status(d) == B.OK
    del ws


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("layer,kw", [
    (ConvLayer("1x1, 16 splits a tile and more", 24, 3, 36, 36, 80, 1, 1, 1, 0), {}),
    (ConvLayer("1x1, an odd element count", 19, 3, 13, 13, 75, 1, 1, 1, 0), dict(dy_layout=B.DY_NPQK, dw_layout=B.DW_KCRS)),
    (ConvLayer("5x5, four channels", 9, 4, 21, 20, 9, 5, 5, 1, 2), dict(x_layout=B.X_NCHW, dy_layout=B.DY_NPQK)),
    (ConvLayer("3x3, 20 channels, odd rows", 5, 20, 9, 11, 20, 3, 3, 1, 1), dict(dy_layout=B.DY_NPQK, dw_layout=B.DW_RSCK)),
], ids=lambda v: v.name if isinstance(v, ConvLayer) else "")
def test_fewer_splits_in_smaller_workspaces(layer, kw, dtype):
    """The FP32-pipe kernel splits as far as the workspace has room for its partial blocks, down to one split; nothing is written beyond it."""
    x, dy = I.make_layer_inputs(layer, dtype, 26, 0)
    ref, dn = oracle.dw_exact(to_f64(x), to_f64(dy), oshape(layer))
    g = GpuLayer(layer, dtype, x, dy, algo=B.ALGO_DIRECT, **kw)
    full, out = B.gaconv_workspace_size(g.desc, B.METHOD_EXACT), layer.k * layer.c * layer.r * layer.s * 4
    copy = g.dy.numel() * g.dy.element_size() if kw.get("dy_layout") == B.DY_NPQK else 0
    least = 17 * 1024 + copy               # (control words and a ragged end)
    assert full > least + 4 * out
    ws, before = torch.empty(full + 4096, dtype=torch.uint8, device="cuda"), None
    for size in (full, full - 16, least + 4 * out, least + 2 * out, least + out, least):
        ws.fill_(0x5a)
        B.gaconv_workspace_init(ws, size)
        g.desc.workspace, g.desc.workspace_bytes = ws.data_ptr(), size
        got = g.exact()
        assert norm_err(got, ref, dn) <= TOL_F32, size
        assert bool((ws[size:] == 0x5a).all()), size
        assert any("direct_tiled_kernel" in n for n in kernel_names(lambda: B.gaconv_dw_exact(g.x, g.dy, g.dw, g.desc)))
    g.desc.workspace_bytes = 16 * 1024 + copy
    with pytest.raises(B.GaconvError) as e:
        B.gaconv_dw_exact(g.x, g.dy, g.dw, g.desc)
    assert e.value.status == B.ERR_WORKSPACE_TOO_SMALL


def test_static_scratch_full_of_a_transposed_gradient():
    """A channels-last gradient of 8.3 MB that is transposed into the built-in array: the partial blocks take what is left."""
    layer = ConvLayer("1x1", 164, 3, 13, 13, 75, 1, 1, 1, 0)
    x, dy = I.make_layer_inputs(layer, torch.float32, 27, 0)
    ref, dn = oracle.dw_exact(to_f64(x), to_f64(dy), oshape(layer))
    g = GpuLayer(layer, torch.float32, x, dy, dy_layout=B.DY_NPQK)
    bare = B.make_desc(layer, torch.float32, dy_layout=B.DY_NPQK)
    assert B.gaconv_workspace_size(bare, B.METHOD_EXACT) > B.gaconv_static_scratch_bytes()
    B.gaconv_dw_exact_static(g.x, g.dy, g.dw, bare)
    assert norm_err(g.logical_dw(), ref, dn) <= TOL_F32 and B.gaconv_poll_async_status_static() == B.OK
