"""The kernels that a call enqueues, from a stream capture of it (CUDA driver API)."""
import ctypes as C

import torch

_RELAXED, _KERNEL = 2, 0          # capture mode; graph node type


class _KernelParams(C.Structure):
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("shared", C.c_uint),
                ("params", C.POINTER(C.c_void_p)), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]


def _cu():
    return C.CDLL("libcuda.so.1")


def _ok(rc):
    assert rc == 0, "CUDA driver error %d" % rc


def captured_kernels(call):
    """[(name, [parameter addresses on the host])] of the kernels that call(stream)
    enqueues, in the order of their creation.  Nothing runs.  The second value
    must be kept while the parameters are read: it holds the graph."""
    cu, s = _cu(), torch.cuda.Stream()
    torch.cuda.synchronize()
    _ok(cu.cuStreamBeginCapture_v2(C.c_void_p(s.cuda_stream), _RELAXED))
    graph = C.c_void_p()
    try:
        with torch.cuda.stream(s):
            call(s)
    finally:
        _ok(cu.cuStreamEndCapture(C.c_void_p(s.cuda_stream), C.byref(graph)))
    n = C.c_size_t()
    _ok(cu.cuGraphGetNodes(graph, None, C.byref(n)))
    nodes = (C.c_void_p * n.value)()
    _ok(cu.cuGraphGetNodes(graph, nodes, C.byref(n)))
    out = []
    for node in nodes:
        kind = C.c_int()
        _ok(cu.cuGraphNodeGetType(C.c_void_p(node), C.byref(kind)))
        if kind.value != _KERNEL:
            continue
        p, name = _KernelParams(), C.c_char_p()
        _ok(cu.cuGraphKernelNodeGetParams_v2(C.c_void_p(node), C.byref(p)))
        if p.func:
            _ok(cu.cuFuncGetName(C.byref(name), C.c_void_p(p.func)))
        else:
            _ok(cu.cuKernelGetName(C.byref(name), C.c_void_p(p.kern)))
        out.append((name.value.decode(), p.params))
    return out, graph


def pointer_param(params, k):
    """The device address that is parameter k of a captured kernel."""
    return C.cast(params[k], C.POINTER(C.c_uint64))[0]


def poke(address, data: bytes):
    """Write bytes to device memory."""
    torch.cuda.synchronize()
    _ok(_cu().cuMemcpyHtoD_v2(C.c_uint64(address), C.c_char_p(data), C.c_size_t(len(data))))
