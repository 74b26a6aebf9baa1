"""The kernels that a call enqueues, read from a stream capture of it: names, grids, blocks and cluster sizes."""
from __future__ import annotations

import ctypes as C

import torch


class _KernelParams(C.Structure):   # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("smem", C.c_uint),
                ("args", C.c_void_p), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]


def kernels(call):
    """[(name, grid, block, CTAs of a cluster)] of call(), which runs once outside the capture and once inside."""
    cu = C.CDLL("libcuda.so.1")

    def check(r):
        assert r == 0, r

    call()
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    graph = C.c_void_p()
    with torch.cuda.stream(stream):
        h = C.c_void_p(stream.cuda_stream)
        check(cu.cuStreamBeginCapture_v2(h, 1))   # thread-local
        try:
            call()
        finally:
            check(cu.cuStreamEndCapture(h, C.byref(graph)))
    count = C.c_size_t()
    check(cu.cuGraphGetNodes(graph, None, C.byref(count)))
    nodes = (C.c_void_p * count.value)()
    check(cu.cuGraphGetNodes(graph, nodes, C.byref(count)))
    out = []
    for node in nodes:
        kind = C.c_int()
        check(cu.cuGraphNodeGetType(C.c_void_p(node), C.byref(kind)))
        if kind.value != 0:   # not a kernel
            continue
        p = _KernelParams()
        check(cu.cuGraphKernelNodeGetParams_v2(C.c_void_p(node), C.byref(p)))
        name = C.c_char_p()
        if p.func:
            check(cu.cuFuncGetName(C.byref(name), C.c_void_p(p.func)))
        else:
            check(cu.cuKernelGetName(C.byref(name), C.c_void_p(p.kern)))
        attr = (C.c_uint * 16)()   # CUlaunchAttributeValue
        check(cu.cuGraphKernelNodeGetAttribute(C.c_void_p(node), 4, attr))   # cluster dimension
        out.append((name.value.decode(), tuple(p.grid), tuple(p.block), max(1, attr[0] * attr[1] * attr[2])))
    check(cu.cuGraphDestroy(graph))
    return out
