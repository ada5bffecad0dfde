"""The kernel launches of a call as (name, grid, block, shared memory), read from a stream capture.

The capture is thrown away: nothing runs.  Names and shapes come from the driver's graph nodes.
"""
import ctypes

import torch


class _KernelNode(ctypes.Structure):
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("smem", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def _ok(rc: int, what: str) -> None:
    assert rc == 0, f"{what}: driver error {rc}"


def captured(call) -> list[tuple[str, int, int, int]]:
    """The launches of call(stream), in no promised order."""
    cu = ctypes.CDLL("libcuda.so.1")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph, s = ctypes.c_void_p(), ctypes.c_void_p(stream.cuda_stream)
    _ok(cu.cuStreamBeginCapture_v2(s, 2), "begin capture")
    try:
        call(stream)
    finally:
        rc = cu.cuStreamEndCapture(s, ctypes.byref(graph))
    _ok(rc, "end capture")
    n = ctypes.c_size_t()
    _ok(cu.cuGraphGetNodes(graph, None, ctypes.byref(n)), "count nodes")
    nodes = (ctypes.c_void_p * n.value)()
    _ok(cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)), "list nodes")
    out = []
    for node in nodes:
        kind = ctypes.c_int()
        _ok(cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)), "node type")
        if kind.value != 0:  # not a kernel
            continue
        k, name = _KernelNode(), ctypes.c_char_p()
        _ok(cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(k)), "kernel node")
        get = (cu.cuFuncGetName, k.func) if k.func else (cu.cuKernelGetName, k.kern)
        _ok(get[0](ctypes.byref(name), ctypes.c_void_p(get[1])), "kernel name")
        out.append((name.value.decode(), k.grid[0], k.block[0], k.smem))
    _ok(cu.cuGraphDestroy(graph), "destroy")
    return out
