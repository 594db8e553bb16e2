"""The channels-last tensor-core kernel (csrc/cl.cu) at the edges of its tiles, against the oracle: odd maps, channel
counts off every tile size, strides, every packing path, several images per chunk, one split and many."""
import re
import threading

import numpy as np
import pytest
import torch

from oracle import oracle
from paper_1908_05460_b200 import binding as B
from paper_1908_05460_b200 import inputs as I
from paper_1908_05460_b200.layers import ConvLayer
from helpers import GpuLayer, kernel_names, norm_err, oshape, to_f64, TOL_F32

pytestmark = pytest.mark.gpu

# (no other tensor-core kernel tiles these maps; each has more products than the kernel is used from, in both types)
SHAPES = [
    ConvLayer("13x11 c19 k87", 15, 19, 13, 11, 87, 3, 3, 1, 1, dy_std=1.0),
    ConvLayer("28x20 c72 k120", 3, 72, 28, 20, 120, 3, 3, 1, 1),
    ConvLayer("7x7 maps, several images, c130 k260", 9, 130, 7, 7, 260, 3, 3, 1, 1),
    ConvLayer("9x24 row pairs, odd rows", 4, 64, 9, 24, 64, 3, 3, 1, 1),
    ConvLayer("stride 2, 27x27 -> 14x14", 4, 64, 27, 27, 100, 3, 3, 2, 1),
    ConvLayer("stride 2, no padding, 5x5", 8, 40, 21, 17, 48, 5, 5, 2, 0),
    ConvLayer("7x7 filter, stride 2, 3 channels", 11, 3, 33, 31, 64, 7, 7, 2, 3),
    ConvLayer("7x7 filter c33", 2, 33, 19, 12, 30, 7, 7, 1, 3),
    ConvLayer("1x1 c200 k72", 7, 200, 11, 5, 72, 1, 1, 1, 0),
    ConvLayer("many splits, k8", 60, 20, 25, 19, 8, 3, 3, 1, 1),
    ConvLayer("one output channel", 102, 48, 31, 15, 1, 3, 3, 1, 1),
    ConvLayer("5x3 maps, more tiles than SMs", 3, 400, 5, 3, 530, 3, 3, 1, 1),
    ConvLayer("3x5 filter", 6, 36, 18, 18, 44, 3, 5, 1, 1),
    ConvLayer("stacked filter rows, 5x5, two row tiles", 12, 72, 17, 11, 40, 5, 5, 1, 2),
    ConvLayer("13 outputs, no padding", 30, 100, 12, 9, 13, 3, 3, 1, 0),
    ConvLayer("stacked filter rows, (pixel, image) order, odd pixels", 30, 130, 5, 9, 40, 5, 5, 1, 2),
    ConvLayer("7x3 filter", 9, 70, 12, 16, 64, 7, 3, 1, 1),
    ConvLayer("odd pixels past a tile, 3 and 70 channels", 15, 3, 33, 35, 70, 3, 3, 1, 1),
    ConvLayer("odd pixels, 24 and 12 channels", 9, 24, 21, 15, 12, 5, 5, 1, 2),
    ConvLayer("stride 2, MMAs of two column shifts and of one", 6, 70, 23, 19, 130, 3, 3, 2, 1),
    ConvLayer("stride 3, 7x7: three shifts, two and two", 12, 30, 30, 25, 100, 7, 7, 3, 3),
    ConvLayer("5x5, tiles of 32 of 72 channels", 5, 72, 15, 15, 136, 5, 5, 1, 2),
    ConvLayer("7x7, tiles of 16 of 70 channels", 6, 70, 13, 10, 131, 7, 7, 1, 3),
    ConvLayer("3 channels, 5x5, rows of 40", 8, 3, 33, 40, 70, 5, 5, 1, 2),
    ConvLayer("4 channels, 3x7, padding on one side", 13, 4, 21, 19, 100, 3, 7, 1, 2),
    ConvLayer("windows of two channels, 9 rows in two tiles", 22, 2, 30, 17, 130, 9, 3, 1, 1),
    ConvLayer("windows of two channels, 7x7, odd rows", 30, 2, 34, 31, 48, 7, 7, 1, 3),
    ConvLayer("3x1 filter, 20 channels", 30, 20, 26, 16, 60, 3, 1, 1, 0),
    ConvLayer("windows of three channels, 5x5, rows of 41", 8, 3, 33, 41, 70, 5, 5, 1, 2),
    # (the gain of gathered windows is a tenth of the estimate without the packing pass of dY, less of it with)
    ConvLayer("windows of two channels, 224 outputs, rows of 43", 19, 2, 43, 43, 224, 3, 3, 1, 1),
    ConvLayer("windows of four channels, 248 outputs, rows of 14", 18, 4, 14, 14, 248, 5, 5, 1, 2),
]
LAYOUTS = {"paper": {}, "nchw": dict(x_layout=B.X_NCHW, dw_layout=B.DW_KCRS),
           "nhwc": dict(dy_layout=B.DY_NPQK, dw_layout=B.DW_KCRS), "rsck": dict(x_layout=B.X_NCHW, dy_layout=B.DY_NPQK, dw_layout=B.DW_RSCK)}


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("li", range(len(SHAPES)), ids=[l.name for l in SHAPES])
def test_every_layout_matches_the_oracle(li, dtype):
    layer = SHAPES[li]
    x, dy = I.make_layer_inputs(layer, dtype, 11, li)
    ref, dn = oracle.dw_exact(to_f64(x), to_f64(dy), oshape(layer), 0.5)
    first = {}
    for name, kw in LAYOUTS.items():
        g = GpuLayer(layer, dtype, x, dy, alpha=0.5, **kw)
        before = B.gaconv_launch_count()
        got = g.exact()
        assert B.gaconv_launch_count() - before <= 3, name
        names = kernel_names(lambda: B.gaconv_dw_exact(g.x, g.dy, g.dw, g.desc))
        assert any("cl_kernel" in k for k in names), name
        if layer.name.startswith("windows"):
            assert any(re.search("pack_kernelI[ft]Lb1E", k) for k in names), (name, names)
        assert norm_err(got, ref, dn) <= TOL_F32 / 2, name        # bf16 products are exact in fp32 as well
        np.testing.assert_array_equal(got, g.exact())
        # the same operands, however they were handed over; only a bf16 gradient on rows of whole 16-byte pieces is read as it
        # lies, so that its pixels are summed in another order when it comes channels last
        order = kw.get("dy_layout", B.DY_NKPQ) if dtype == torch.bfloat16 and layer.q % 8 == 0 else None
        np.testing.assert_array_equal(got, first.setdefault(order, got))
        assert B.gaconv_poll_async_status(g.desc) == B.OK
    few = GpuLayer(layer, dtype, x, dy, alpha=0.5, sm_budget=11)
    assert norm_err(few.exact(), ref, dn) <= TOL_F32 / 2


def test_long_sums_keep_fp32_accuracy():
    """Tens of thousands of products per output and an activation with a mean: the tensor core's own additions truncate,
    so without the periodic hand-over to fp32 registers the error would grow with the sum."""
    layer = ConvLayer("long", 40, 16, 45, 47, 16, 3, 3, 1, 1, dy_std=1.0)
    for dtype in (torch.float32, torch.bfloat16):
        x, dy = I.make_layer_inputs(layer, dtype, 11, 50)
        dy = (dy.float() + 0.5).to(dtype)
        ref, dn = oracle.dw_exact(to_f64(x), to_f64(dy), oshape(layer))
        g = GpuLayer(layer, dtype, x, dy, sm_budget=2)
        assert norm_err(g.exact(), ref, dn) <= 2e-6


def test_static_scratch_takes_the_kernels_that_fit():
    """Scratch beyond the built-in array: gaconv_dw_exact_static falls back to the kernels that need less of it."""
    layer = ConvLayer("packed copies of 12 MB", 40, 64, 30, 30, 64, 3, 3, 1, 1)
    x, dy = I.make_layer_inputs(layer, torch.float32, 11, 51)
    g = GpuLayer(layer, torch.float32, x, dy)
    want = g.exact()
    bare = B.make_desc(layer, torch.float32)
    assert B.gaconv_workspace_size(bare, B.METHOD_EXACT) > B.gaconv_static_scratch_bytes()
    g.dw.fill_(float("nan"))
    B.gaconv_dw_exact_static(g.x, g.dy, g.dw, bare)
    got = g.logical_dw()
    assert np.max(np.abs(got - want)) <= 1e-4 * np.abs(want).max() and B.gaconv_poll_async_status_static() == B.OK


@pytest.mark.parametrize("layer,kw", [
    (ConvLayer("windows of three channels", 93, 3, 49, 49, 48, 3, 3, 1, 1), {}),
    (ConvLayer("windows of a 7x7 filter", 300, 3, 25, 25, 32, 7, 7, 1, 3), dict(x_layout=B.X_NCHW, sm_budget=18)),
    (ConvLayer("5x5 on 3x3 maps, blocks of 5 MB", 979, 200, 3, 3, 112, 5, 5, 1, 1), dict(x_layout=B.X_NCHW)),
], ids=lambda v: v.name if isinstance(v, ConvLayer) else "")
def test_static_scratch_without_room_for_the_first_plan(layer, kw):
    """What the planner likes best (gathered windows, more splits) is beyond the built-in array, and the other kernels would have to transpose
    operands that are, too: the channels-last kernel in less scratch."""
    x, dy = I.make_layer_inputs(layer, torch.bfloat16, 25, 0)
    g = GpuLayer(layer, torch.bfloat16, x, dy, dy_layout=B.DY_NPQK, **kw)
    bare = B.make_desc(layer, torch.bfloat16, dy_layout=B.DY_NPQK, **kw)
    assert B.gaconv_workspace_size(bare, B.METHOD_EXACT) > B.gaconv_static_scratch_bytes()
    want = g.exact()
    g.dw.fill_(float("nan"))
    B.gaconv_dw_exact_static(g.x, g.dy, g.dw, bare)
    got = g.logical_dw()
    assert B.gaconv_poll_async_status_static() == B.OK
    assert any("cl_kernel" in k for k in kernel_names(lambda: B.gaconv_dw_exact_static(g.x, g.dy, g.dw, bare)))
    xd, dyd, rng = to_f64(x), to_f64(dy), np.random.default_rng(4)
    for k, c, r, s in zip(*(rng.integers(0, m, 60).tolist() for m in (layer.k, layer.c, layer.r, layer.s))):
        v, norm = oracle.dw_exact_at(xd, dyd, oshape(layer), k, c, r, s)
        assert abs(got[k, c, r, s] - v) <= TOL_F32 * norm and abs(want[k, c, r, s] - v) <= TOL_F32 * norm
    assert np.all(np.isfinite(got))


# strides and boxes beyond what a tensor map steps over (8 pixels, 256 a side): other kernels take them
FAR = [
    ConvLayer("stride 9", 20, 64, 40, 37, 96, 3, 3, 9, 1),
    ConvLayer("stride 12, 12x12 patches", 8, 3, 60, 48, 200, 12, 12, 12, 0),
    ConvLayer("stride 9, 8x8 outputs", 2, 16, 72, 72, 16, 3, 3, 9, 1),
    ConvLayer("stride 8, the largest step", 20, 64, 40, 37, 96, 3, 3, 8, 1),
    ConvLayer("stride 5, rows of 64 outputs", 2, 16, 20, 320, 16, 3, 3, 5, 1),
    ConvLayer("stride 5, 64 rows of one output", 2, 16, 320, 1, 16, 1, 1, 5, 0),
]


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("li", range(len(FAR)), ids=[l.name for l in FAR])
def test_large_strides(li, dtype):
    layer = FAR[li]
    x, dy = I.make_layer_inputs(layer, dtype, 16, li)
    ref, dn = oracle.dw_exact(to_f64(x), to_f64(dy), oshape(layer), 0.5)
    for name, kw in LAYOUTS.items():
        g = GpuLayer(layer, dtype, x, dy, alpha=0.5, **kw)
        assert norm_err(g.exact(), ref, dn) <= TOL_F32, name
        assert B.gaconv_poll_async_status(g.desc) == B.OK
        if li in (0, 3):
            names = kernel_names(lambda: B.gaconv_dw_exact(g.x, g.dy, g.dw, g.desc))
            assert any("cl_kernel" in k for k in names) == (layer.stride <= 8), names


def _without_padding(x, dy, layer, k):
    """dW[k] with the products of the padding left out (they are zeros unless dY is not finite there)."""
    l, out = layer, np.zeros((layer.c, layer.r, layer.s))
    for r in range(l.r):
        for s in range(l.s):
            ps = [p for p in range(l.p) if 0 <= p * l.stride + r - l.pad < l.h]
            qs = [q for q in range(l.q) if 0 <= q * l.stride + s - l.pad < l.w]
            xs = x[:, :, [p * l.stride + r - l.pad for p in ps]][:, :, :, [q * l.stride + s - l.pad for q in qs]]
            out[:, r, s] = (xs * dy[:, k:k + 1][:, :, ps][:, :, :, qs]).sum(axis=(0, 2, 3))
    return out


def _alike(got, ref, bound):
    with np.errstate(invalid="ignore"):
        return (np.isnan(got) & np.isnan(ref)) | (got == ref) | (np.abs(got - ref) <= bound)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("li", range(len(SHAPES)), ids=[l.name for l in SHAPES])
def test_values_that_are_not_finite(li, dtype):
    """Infinities and NaNs reach the elements that they are part of, and no others; an infinite product stays infinite."""
    layer = SHAPES[li]
    l = layer
    x, dy = I.make_layer_inputs(layer, dtype, 18, li)
    inf, nan = float("inf"), float("nan")
    x[0, 0, 0, 0], x[1, l.c // 2, l.h - 1, l.w - 1], x[l.n - 1, l.c - 1, l.h // 2, l.w // 2] = inf, -inf, nan
    if l.k > 2:
        dy[0, 0, l.p // 2, l.q // 2], dy[l.n - 1, l.k // 2, 0, 0], dy[1, l.k - 1, l.p - 1, l.q - 1] = inf, -inf, nan
    xd, dyd = to_f64(x), to_f64(dy)
    with np.errstate(invalid="ignore"):
        ref, _ = oracle.dw_exact(xd, dyd, oshape(layer), 0.5)
        bare = ref.copy()
        for k in {0, l.k // 2, l.k - 1}:
            bare[k] = 0.5 * _without_padding(xd, dyd, layer, k)
        _, dn = oracle.dw_exact(np.where(np.isfinite(xd), xd, 0.0), np.where(np.isfinite(dyd), dyd, 0.0), oshape(layer), 0.5)
    assert np.isinf(ref).any() and np.isnan(ref).any()
    for kw in (LAYOUTS["paper"], LAYOUTS["rsck"], dict(sm_budget=1), dict(LAYOUTS["nchw"], sm_budget=1)):       # (one SM: one split)
        g = GpuLayer(layer, dtype, x, dy, alpha=0.5, **kw)
        got = g.exact()
        ok = _alike(got, ref, TOL_F32 * dn) | _alike(got, bare, TOL_F32 * dn)
        assert ok.all(), (kw, int((~ok).sum()), np.argwhere(~ok)[:3].tolist())
        np.testing.assert_array_equal(got, g.exact())


@pytest.mark.parametrize("method", ["exact", "host", "top1"])
@pytest.mark.parametrize("layer,dtype,kw", [
    (ConvLayer("packed planes", 24, 64, 30, 30, 64, 3, 3, 1, 1), torch.float32, {}),
    (ConvLayer("packed gradient", 20, 72, 28, 20, 120, 3, 3, 1, 1), torch.bfloat16, {}),
    (ConvLayer("packed, channels first", 20, 72, 28, 20, 120, 3, 3, 1, 1), torch.bfloat16, dict(x_layout=B.X_NCHW)),
    (ConvLayer("packed windows", 20, 3, 33, 31, 48, 7, 7, 1, 3), torch.bfloat16, dict(x_layout=B.X_NCHW, dy_layout=B.DY_NPQK)),
    (ConvLayer("packed windows of fp32", 40, 4, 29, 30, 40, 3, 3, 1, 1), torch.float32, dict(dy_layout=B.DY_NPQK)),
    (ConvLayer("top-1 by the dense route", 20, 256, 8, 8, 100, 3, 3, 1, 1), torch.bfloat16, dict(x_layout=B.X_NCHW, dy_layout=B.DY_NPQK)),
], ids=lambda v: v.name if isinstance(v, ConvLayer) else None)
def test_smaller_workspaces(layer, dtype, kw, method):
    """Without room for packed operands the older kernels take the call; what is accepted stays within the bytes it was given."""
    x, dy = I.make_layer_inputs(layer, dtype, 19, 0)
    ref, dn = oracle.dw_top1(to_f64(x), to_f64(dy), oshape(layer)) if method == "top1" else oracle.dw_exact(to_f64(x), to_f64(dy), oshape(layer))
    tol = 2.0 ** -8 + 1e-4 if method == "top1" and dtype == torch.bfloat16 else TOL_F32          # (the dense route rounds a map's sum once)
    g = GpuLayer(layer, dtype, x, dy, **kw)
    which = {"exact": B.METHOD_EXACT, "host": B.METHOD_EXACT, "top1": B.METHOD_TOP1}[method]
    full, accepted = B.gaconv_workspace_size(g.desc, which), []
    x_host, dy_host, dw_host = g.x.cpu().pin_memory(), g.dy.cpu().pin_memory(), g.dw.cpu().pin_memory()
    ws = torch.empty(full + 4096, dtype=torch.uint8, device="cuda")
    for size in [full, full - 16] + [max(17024, full * i // 32) for i in range(30, 0, -3)]:
        ws.fill_(0x5a)
        B.gaconv_workspace_init(ws, size)
        g.desc.workspace, g.desc.workspace_bytes = ws.data_ptr(), size
        try:
            if method == "host":
                dw_host.fill_(float("nan"))
                B.gaconv_dw_from_host(B.METHOD_EXACT, x_host, dy_host, dw_host, g.x, g.dy, g.dw, g.desc)
                got = g.logical_dw()
                np.testing.assert_array_equal(dw_host.numpy(), g.dw.cpu().numpy())
            else:
                got = g.exact() if method == "exact" else g.approx(B.METHOD_TOP1)
        except B.GaconvError as e:
            assert e.status == B.ERR_WORKSPACE_TOO_SMALL
            continue
        assert norm_err(got, ref, dn) <= tol
        assert bool((ws[size:] == 0x5a).all()), size
        assert B.gaconv_poll_async_status(g.desc) == B.OK
        accepted.append(size)
    assert accepted[0] == full
    if method != "top1" and "packed" in layer.name:
        assert len(accepted) > 1, (full, accepted)


def test_packed_rows_tight_and_spread():
    """A packed bf16 gradient of 120 channels on rows of 128, or without gaps where the workspace has no room for those: the same bits."""
    layer = ConvLayer("28x20", 6, 72, 28, 20, 120, 3, 3, 1, 1)
    x, dy = I.make_layer_inputs(layer, torch.bfloat16, 23, 0)
    g = GpuLayer(layer, torch.bfloat16, x, dy, x_layout=B.X_NCHW)
    want, full = g.exact(), B.gaconv_workspace_size(g.desc, B.METHOD_EXACT)
    ref, dn = oracle.dw_exact(to_f64(x), to_f64(dy), oshape(layer))
    assert norm_err(want, ref, dn) <= TOL_F32 / 2
    tight = full - 6 * 28 * 20 * (128 - 120) * 2
    for size, kernel in ((full, "cl_kernel"), (full - 16, "cl_kernel"), (tight, "cl_kernel"), (tight - 16, "direct_tiled_kernel")):
        g.desc.workspace_bytes = size
        assert any(kernel in n for n in kernel_names(lambda: B.gaconv_dw_exact(g.x, g.dy, g.dw, g.desc))), size
        got = g.exact()
        assert norm_err(got, ref, dn) <= TOL_F32
        if kernel == "cl_kernel":
            np.testing.assert_array_equal(got, want)


@pytest.mark.parametrize("layer,dtype,kernel", [
    (ConvLayer("channels last, nothing packed", 4, 64, 9, 24, 64, 3, 3, 1, 1), torch.bfloat16, "cl_kernel"),
    (ConvLayer("older tensor-core kernel", 8, 16, 32, 32, 16, 3, 3, 1, 1), torch.bfloat16, "exact_tc_kernel"),
    (ConvLayer("mma.sync", 6, 16, 32, 32, 16, 3, 3, 1, 1), torch.float32, "direct_mma_kernel"),
    (ConvLayer("stem", 5, 3, 32, 32, 16, 3, 3, 1, 1), torch.float32, "stem_mma_kernel"),
], ids=lambda v: v.name if isinstance(v, ConvLayer) else "")
def test_first_call_of_a_thread(layer, dtype, kernel):
    """A thread that has not touched the GPU yet, so that it has no context when the tensor maps are made."""
    c = GpuLayer(layer, dtype, *I.make_layer_inputs(layer, dtype, 20, 0))
    alone, errors, stream = c.exact(), [], torch.cuda.Stream().cuda_stream
    assert any(kernel in k for k in kernel_names(lambda: B.gaconv_dw_exact(c.x, c.dy, c.dw, c.desc)))
    c.dw.fill_(float("nan"))
    torch.cuda.synchronize()

    def work():
        try:
            B.gaconv_dw_exact(c.x, c.dy, c.dw, c.desc, stream)
        except B.GaconvError as e:
            errors.append(e)

    t = threading.Thread(target=work)
    t.start()
    t.join()
    assert not errors, errors[0]
    np.testing.assert_array_equal(c.logical_dw(), alone)


def test_threads_with_layers_of_one_kernel_and_different_shared_memory():
    """Two threads on streams of their own; the layers take the same instance of the kernel with 97 and with 217 KB of shared memory."""
    layers = [ConvLayer("97 KB", 4, 64, 9, 24, 64, 3, 3, 1, 1), ConvLayer("217 KB", 9, 70, 12, 16, 64, 7, 3, 1, 1)]
    calls = [GpuLayer(l, torch.bfloat16, *I.make_layer_inputs(l, torch.bfloat16, 20, i)) for i, l in enumerate(layers)]
    alone = [c.exact() for c in calls]
    names = [next(k for k in kernel_names(lambda: B.gaconv_dw_exact(c.x, c.dy, c.dw, c.desc)) if "cl_kernel" in k) for c in calls]
    assert names[0] == names[1]
    errors = []

    def work(c, stream):
        try:
            for _ in range(4000):
                B.gaconv_dw_exact(c.x, c.dy, c.dw, c.desc, stream)
        except B.GaconvError as e:
            errors.append(e)

    threads = [threading.Thread(target=work, args=(c, torch.cuda.Stream())) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
    for c, want in zip(calls, alone):
        np.testing.assert_array_equal(c.logical_dw(), want)


@pytest.mark.parametrize("layer,budget,kernel", [
    (ConvLayer("5x5, 40 channels", 16, 40, 16, 16, 64, 5, 5, 1, 2), 0, "cl_kernel"),
    (ConvLayer("5x5, 64 channels", 16, 64, 16, 16, 64, 5, 5, 1, 2), 0, "exact_tc_kernel"),
    (ConvLayer("5x5, 64 channels, 88 outputs", 16, 64, 16, 16, 88, 5, 5, 1, 2), 0, "exact_tc_kernel"),
    (ConvLayer("5x5, 64 channels, 96 outputs", 16, 64, 16, 16, 96, 5, 5, 1, 2), 0, "cl_kernel"),
    (ConvLayer("7x7, 64 channels, 128 outputs", 16, 64, 16, 16, 128, 7, 7, 1, 3), 0, "exact_tc_kernel"),
    (ConvLayer("7x7, 24 channels on 32x32", 9, 24, 32, 32, 16, 7, 7, 1, 3), 0, "cl_kernel"),
    (ConvLayer("stem of 64 outputs, 256 images", 256, 3, 32, 32, 64, 3, 3, 1, 1), 0, "cl_kernel"),
    (ConvLayer("stem of 64 outputs, 64 images", 64, 3, 32, 32, 64, 3, 3, 1, 1), 0, "stem_mma_kernel"),
    (ConvLayer("stem of 64 outputs, 64 images, few SMs", 64, 3, 32, 32, 64, 3, 3, 1, 1), 37, "cl_kernel"),
    (ConvLayer("stem of 16 outputs, few SMs", 128, 3, 32, 32, 16, 3, 3, 1, 1), 18, "stem_mma_kernel"),
    (ConvLayer("5x5 stem, 64 images", 64, 3, 32, 32, 64, 5, 5, 1, 2), 0, "cl_kernel"),
    (ConvLayer("a large dW with short sums", 64, 256, 8, 8, 256, 3, 3, 1, 1), 0, "exact_tc_kernel"),
    (ConvLayer("a large dW past the line", 96, 256, 8, 8, 256, 3, 3, 1, 1), 0, "cl_kernel"),
    (ConvLayer("64 channels on few SMs", 32, 64, 8, 8, 64, 3, 3, 1, 1), 18, "exact_tc_kernel"),
    (ConvLayer("64 channels on few SMs, stride 2", 32, 64, 16, 16, 64, 3, 3, 2, 1), 18, "cl_kernel"),
    (ConvLayer("64 channels on few SMs, 450 images", 450, 64, 8, 8, 64, 3, 3, 1, 1), 18, "cl_kernel"),
], ids=lambda v: v.name if isinstance(v, ConvLayer) else str(v))
def test_either_side_of_a_line(layer, budget, kernel):
    """bf16 layers that both tensor-core kernels can do, around the lines between them: the kernel, and its results on samples."""
    x, dy = I.make_layer_inputs(layer, torch.bfloat16, 21, 0)
    g = GpuLayer(layer, torch.bfloat16, x, dy, sm_budget=budget)
    names = kernel_names(lambda: B.gaconv_dw_exact(g.x, g.dy, g.dw, g.desc))
    assert any(kernel in n for n in names), names
    got, xd, dyd = g.exact(), to_f64(x), to_f64(dy)
    rng = np.random.default_rng(3)
    for k, c, r, s in zip(*(rng.integers(0, m, 60).tolist() for m in (layer.k, layer.c, layer.r, layer.s))):
        v, norm = oracle.dw_exact_at(xd, dyd, oshape(layer), k, c, r, s)
        assert abs(got[k, c, r, s] - v) <= TOL_F32 * norm
    assert np.all(np.isfinite(got)) and B.gaconv_poll_async_status(g.desc) == B.OK


@pytest.mark.parametrize("layer,dtype,budget,kernel", [
    (ConvLayer("5x5, stride 2", 60, 3, 64, 64, 40, 5, 5, 2, 2), torch.bfloat16, 18, "stem_mma_kernel"),
    (ConvLayer("5x5, stride 2, one channel", 50, 1, 96, 96, 128, 5, 5, 2, 2), torch.bfloat16, 0, "stem_mma_kernel"),
    (ConvLayer("5x5, windows", 60, 3, 32, 32, 40, 5, 5, 1, 2), torch.bfloat16, 18, "cl_kernel"),
    (ConvLayer("3x3, 16 outputs", 220, 1, 96, 96, 16, 3, 3, 1, 1), torch.bfloat16, 0, "stem_mma_kernel"),
    (ConvLayer("5x5, stride 2", 70, 3, 64, 64, 64, 5, 5, 2, 2), torch.float32, 0, "stem_mma_kernel"),
    (ConvLayer("5x5, windows of two channels", 30, 2, 48, 48, 96, 5, 5, 1, 2), torch.float32, 0, "stem_mma_kernel"),
    (ConvLayer("5x5, 48 outputs", 60, 3, 32, 32, 48, 5, 5, 1, 2), torch.float32, 0, "stem_mma_kernel"),
    (ConvLayer("5x5, 64 outputs", 60, 3, 32, 32, 64, 5, 5, 1, 2), torch.float32, 0, "cl_kernel"),
], ids=lambda v: v.name if isinstance(v, ConvLayer) else str(v))
def test_stems_either_side_of_a_line(layer, dtype, budget, kernel):
    """Image stems that both kernels can do: the plain form of the channels-last kernel, and its six products where few columns are in use, are slower."""
    x, dy = I.make_layer_inputs(layer, dtype, 29, 0)
    g = GpuLayer(layer, dtype, x, dy, sm_budget=budget)
    names = kernel_names(lambda: B.gaconv_dw_exact(g.x, g.dy, g.dw, g.desc))
    assert any(kernel in n for n in names), names
    got, xd, dyd = g.exact(), to_f64(x), to_f64(dy)
    rng = np.random.default_rng(5)
    for k, c, r, s in zip(*(rng.integers(0, m, 40).tolist() for m in (layer.k, layer.c, layer.r, layer.s))):
        v, norm = oracle.dw_exact_at(xd, dyd, oshape(layer), k, c, r, s)
        assert abs(got[k, c, r, s] - v) <= TOL_F32 * norm
    assert np.all(np.isfinite(got)) and B.gaconv_poll_async_status(g.desc) == B.OK


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("layer", [
    ConvLayer("two columns, padding 2", 43, 9, 8, 8, 244, 5, 2, 1, 2),
    ConvLayer("2x2 filter, padding 2 on 4x4", 150, 118, 4, 4, 19, 2, 2, 1, 2),
    ConvLayer("3x3 filter, padding 4 on 5x5", 150, 20, 5, 5, 26, 3, 3, 1, 4),
    ConvLayer("rows of one pixel, padding 5", 100, 79, 8, 1, 30, 4, 4, 1, 5),
    ConvLayer("odd rows of eight, 4 outputs", 61, 159, 19, 8, 4, 3, 3, 1, 1),
], ids=lambda l: l.name)
def test_windows_wholly_in_the_padding(layer, dtype):
    """Output pixels that meet no pixel of X, and the last pairs of eight pixels of a band: nothing beyond the tiles is multiplied."""
    x, dy = I.make_layer_inputs(layer, dtype, 22, 0)
    ref, dn = oracle.dw_exact(to_f64(x), to_f64(dy), oshape(layer))
    for kw in (*LAYOUTS.values(), dict(sm_budget=7)):
        g = GpuLayer(layer, dtype, x, dy, **kw)
        assert norm_err(g.exact(), ref, dn) <= TOL_F32, kw
        assert B.gaconv_poll_async_status(g.desc) == B.OK
