"""The kernel launches of a call, read from a captured graph of it."""
import ctypes

KERNEL_NODE = 0


class _KernelNodeParams(ctypes.Structure):      # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("shared", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def launches(call):
    """(grid, block, dynamic shared memory) of every kernel node of the graph
    captured from call(stream).  The call must have run before: the first
    launch of a kernel sets its limits."""
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph, n = ctypes.c_void_p(), ctypes.c_size_t()
    assert cu.cuStreamBeginCapture_v2(ctypes.c_void_p(stream.cuda_stream), 1) == 0   # this thread's
    try:
        call(stream)
    finally:
        ended = cu.cuStreamEndCapture(ctypes.c_void_p(stream.cuda_stream), ctypes.byref(graph))
    assert ended == 0
    try:
        assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
        nodes = (ctypes.c_void_p * n.value)()
        assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
        found = []
        for node in nodes:
            kind, p = ctypes.c_int(), _KernelNodeParams()
            assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
            if kind.value != KERNEL_NODE:
                continue
            assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)) == 0
            found.append((tuple(p.grid), tuple(p.block), p.shared))
        return found
    finally:
        cu.cuGraphDestroy(graph)
