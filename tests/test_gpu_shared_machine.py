"""The older tensor-core kernel with short main loops next to copies of itself: its two issuers take alternate chunks of a ring
with an odd number of stages, copies land late and out of turn, and every result must still be the one of a call on its own."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_1908_05460_b200 import binding as B
from paper_1908_05460_b200 import inputs as I
from paper_1908_05460_b200.layers import ConvLayer
from helpers import GpuLayer, norm_err, oshape, to_f64, TOL_F32

pytestmark = pytest.mark.gpu
LANES, COPIES, ROUNDS = 12, 24, 40


@pytest.mark.parametrize("dtype,layer", [
    (torch.bfloat16, ConvLayer("1x1, three stages", 128, 64, 16, 16, 128, 1, 1, 1, 0)),
    (torch.bfloat16, ConvLayer("3x3, five stages", 64, 64, 8, 8, 64, 3, 3, 1, 1)),
    (torch.float32, ConvLayer("1x1 on split planes, five stages", 24, 64, 16, 16, 48, 1, 1, 1, 0)),
], ids=lambda v: v.name if isinstance(v, ConvLayer) else str(v).split(".")[1])
def test_results_do_not_depend_on_what_runs_beside(dtype, layer):
    calls = []
    for i in range(COPIES):
        x, dy = I.make_layer_inputs(layer, dtype, 17, i % 3)
        calls.append(GpuLayer(layer, dtype, x, dy, algo=B.ALGO_TENSOR, sm_budget=18))
    alone = [c.exact() for c in calls[:3]]                         # synchronised, one after the other
    ref, dn = oracle.dw_exact(to_f64(I.make_layer_inputs(layer, dtype, 17, 0)[0]), to_f64(I.make_layer_inputs(layer, dtype, 17, 0)[1]), oshape(layer))
    assert norm_err(alone[0], ref, dn) <= TOL_F32
    lanes = [torch.cuda.Stream() for _ in range(LANES)]

    def everything():
        main = torch.cuda.current_stream()
        fork = torch.cuda.Event()
        fork.record(main)
        for s in lanes:
            s.wait_event(fork)
        for i, c in enumerate(calls):
            B.gaconv_dw_exact(c.x, c.dy, c.dw, c.desc, lanes[i % LANES])
        for s in lanes:
            join = torch.cuda.Event()
            join.record(s)
            main.wait_event(join)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        everything()
    for _ in range(ROUNDS):
        for c in calls:
            c.dw.fill_(float("nan"))
        graph.replay()
        for i, c in enumerate(calls):
            np.testing.assert_array_equal(c.logical_dw(), alone[i % 3])
    assert all(B.gaconv_poll_async_status(c.desc) == B.OK for c in calls)
