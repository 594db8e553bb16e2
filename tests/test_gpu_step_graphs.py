"""Repeated steps (gaconv_schedule_run_step from its second call with the same buffers on): results are those of the
per-layer calls, whatever the step, the stream, or what else the schedule has run in between."""
import numpy as np
import pytest
import torch

from paper_1908_05460_b200 import binding as B
from paper_1908_05460_b200 import inputs as I
from paper_1908_05460_b200.layers import ConvLayer
from helpers import GpuLayer

pytestmark = pytest.mark.gpu

LAYERS = [ConvLayer("a", 4, 16, 16, 16, 16, 3, 3, 1, 1), ConvLayer("b", 5, 24, 13, 11, 40, 3, 3, 1, 1), ConvLayer("c", 3, 3, 32, 32, 16, 3, 3, 1, 1),
          ConvLayer("d", 6, 64, 8, 8, 64, 3, 3, 1, 1), ConvLayer("e", 40, 30, 9, 9, 56, 3, 3, 1, 1),
          ConvLayer("f", 4, 16, 16, 16, 24, 5, 5, 1, 2)]


def _layers(dtype, dw_layout=B.DW_KRSC):
    return [GpuLayer(l, dtype, *I.make_layer_inputs(l, dtype, 12, i), alpha=0.5, dw_layout=dw_layout) for i, l in enumerate(LAYERS)]


def _per_layer(sched, step, gs):
    out = []
    for i, g in enumerate(gs):
        g.dw.fill_(float("nan"))
        sched.run_layer(i, step, g.x, g.dy, g.dw, g.desc)
        out.append(g.logical_dw())
    return out


@pytest.mark.parametrize("method", [B.METHOD_TOP1, B.METHOD_RANDOM, B.METHOD_ZERO], ids=["top1", "random", "zero"])
@pytest.mark.parametrize("lanes", [1, 4])
def test_repeated_steps_equal_per_layer_calls(method, lanes):
    for dw_layout in (B.DW_KRSC, B.DW_KCRS):                   # the random kernel differs
        gs = _layers(torch.bfloat16, dw_layout)
        sched = B.Schedule(len(gs), B.SCHED_ALT_LAYER_ALT_BATCH, method, seed=77)
        packed = sched.pack_step([g.x for g in gs], [g.dy for g in gs], [g.dw for g in gs], [g.desc for g in gs])
        side = torch.cuda.Stream()
        for step in (1, 1, 1, 3, 0, 5, 0, 0, 2, 7):             # odd steps share their methods but not their seeds
            want = _per_layer(sched, step, gs)
            for g in gs:
                g.dw.fill_(float("nan"))
            torch.cuda.synchronize()
            before = B.gaconv_launch_count()
            with torch.cuda.stream(side if step == 5 else torch.cuda.current_stream()):
                sched.run_step(step, packed, lanes=lanes)
            assert B.gaconv_launch_count() - before >= len(gs)
            for g, w in zip(gs, want):
                np.testing.assert_array_equal(g.logical_dw(), w)
                assert B.gaconv_poll_async_status(g.desc) == B.OK
        sched.close()


def test_other_buffers_and_new_inputs_are_seen():
    sets = [_layers(torch.float32) for _ in range(11)]          # more sets than a schedule keeps recorded steps for
    sched = B.Schedule(len(LAYERS), B.SCHED_EVERY_4TH_LAYER, B.METHOD_TOP1)
    packs = [sched.pack_step([g.x for g in gs], [g.dy for g in gs], [g.dw for g in gs], [g.desc for g in gs]) for gs in sets]
    for rep in range(3):
        for i, (gs, p) in enumerate(zip(sets, packs)):
            for g in gs:
                g.dy.mul_(1.0 + 0.25 * (i + rep))               # the values change in place, as in training
            want = _per_layer(sched, 2, gs)
            for g in gs:
                g.dw.fill_(float("nan"))
            sched.run_step(2, p, lanes=3)
            for g, w in zip(gs, want):
                np.testing.assert_array_equal(g.logical_dw(), w)
    gs = sets[0]
    gs[1].desc.alpha = 2.0                                      # a changed descriptor is another step
    want = _per_layer(sched, 2, gs)
    for _ in range(3):
        sched.run_step(2, packs[0], lanes=3)
        np.testing.assert_array_equal(gs[1].logical_dw(), want[1])
