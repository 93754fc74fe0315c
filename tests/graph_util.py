"""Kernel nodes of a call captured into a CUDA graph (for the GPU tests)."""
import ctypes

import torch


class _Params(ctypes.Structure):  # CUDA_KERNEL_NODE_PARAMS (v2)
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("smem", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def kernel_blocks(call):
    """Threads per block of every kernel node of call(stream), which runs once before it is captured."""
    call(torch.cuda.current_stream())
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call(torch.cuda.current_stream())
    # the driver's calls: the library has a runtime of its own, whose kernels torch's does not know
    cu, graph, n = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(g.raw_cuda_graph()), ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    blocks = []
    for node in nodes:
        kind, p = ctypes.c_int(-1), _Params()
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value == 0:  # a kernel
            assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)) == 0
            blocks.append(p.block[0] * p.block[1] * p.block[2])
    return blocks
