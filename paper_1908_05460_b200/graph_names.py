"""Which kernels a call enqueues, read from a CUDA graph that the call is captured into."""
from __future__ import annotations

import ctypes

import torch


class _KernelNodeParams(ctypes.Structure):
    _fields_ = [("func", ctypes.c_void_p), ("dims", ctypes.c_uint * 7), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def kernel_names(call) -> list[str]:
    """(Mangled) names of the kernels that `call` enqueues on the current stream, read from a graph that it is captured into (and
    that is never launched): what a result cannot tell, namely which kernel it came from."""
    cu = ctypes.CDLL("libcuda.so.1")
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    handle, count = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(handle, None, ctypes.byref(count)) == 0
    nodes = (ctypes.c_void_p * count.value)()
    assert cu.cuGraphGetNodes(handle, nodes, ctypes.byref(count)) == 0
    names = []
    for node in nodes:
        kind, p, name = ctypes.c_int(-1), _KernelNodeParams(), ctypes.c_char_p()
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value != 0:                 # CU_GRAPH_NODE_TYPE_KERNEL
            continue
        assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)) == 0
        get, what = (cu.cuFuncGetName, p.func) if p.func else (cu.cuKernelGetName, p.kern)
        assert get(ctypes.byref(name), ctypes.c_void_p(what)) == 0
        names.append(name.value.decode())
    return names
