"""Kernels that a call would launch, from the stream capture of the call (nothing runs)."""
import ctypes as C

import torch


class _KernelNode(C.Structure):  # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("smem", C.c_uint),
                ("params", C.c_void_p), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]


def _ok(code):
    assert code == 0, f"CUDA driver error {code}"


def kernels(call):
    """[(name, grid, block)] of the kernels that call(stream) launches on that stream, in order."""
    cu = C.CDLL("libcuda.so.1")
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    st, graph = C.c_void_p(stream.cuda_stream), C.c_void_p()
    # CU_STREAM_CAPTURE_MODE_RELAXED: solvers of earlier tests may be collected, and freed, meanwhile
    _ok(cu.cuStreamBeginCapture_v2(st, 2))
    try:
        call(stream)
    finally:
        code = cu.cuStreamEndCapture(st, C.byref(graph))
    _ok(code)
    try:
        n = C.c_size_t()
        _ok(cu.cuGraphGetNodes(graph, None, C.byref(n)))
        nodes = (C.c_void_p * n.value)()
        if n.value:
            _ok(cu.cuGraphGetNodes(graph, nodes, C.byref(n)))
        out = []
        for node in nodes:  # in the order of their creation
            kind = C.c_int()
            _ok(cu.cuGraphNodeGetType(C.c_void_p(node), C.byref(kind)))
            if kind.value != 0:  # CU_GRAPH_NODE_TYPE_KERNEL
                continue
            k, name = _KernelNode(), C.c_char_p()
            _ok(cu.cuGraphKernelNodeGetParams_v2(C.c_void_p(node), C.byref(k)))
            if k.func:
                _ok(cu.cuFuncGetName(C.byref(name), C.c_void_p(k.func)))
            else:
                _ok(cu.cuKernelGetName(C.byref(name), C.c_void_p(k.kern)))
            out.append((name.value.decode(), k.grid[0], k.block[0]))
        return out
    finally:
        _ok(cu.cuGraphDestroy(graph))
