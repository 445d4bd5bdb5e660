"""The kernels that a call launches, read from a CUDA graph captured around it (driver API through ctypes):
which form of a product a call takes, and in how many launches."""
import ctypes
import re

import torch


class _Params(ctypes.Structure):
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("shared", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def _ok(status, what):
    if status != 0:
        raise RuntimeError("%s: CUDA driver status %d" % (what, status))


def _demangle(name):
    """(last name, template arguments) of a mangled function name: _ZN 2aq 39_GLOBAL... 15gemv_lut_kernel ILi0E...E."""
    i, last = (3 if name.startswith("_ZN") else 2), name
    while name[i:i + 1].isdigit():
        m = re.match(r"\d+", name[i:])
        i += m.end()
        last = name[i:i + int(m.group())]
        i += int(m.group())
    m = re.match(r"I((?:L[a-z]\d+E)+)E", name[i:])
    return last, tuple(int(v) for v in re.findall(r"L[a-z](\d+)E", m.group(1))) if m else ()


def kernels(call):
    """[(name, template arguments, grid, block, cluster size)] of the kernels that call() enqueues on the current
    stream, in the order of their nodes. call() runs once beforehand, so that workspaces exist."""
    cu = ctypes.CDLL("libcuda.so.1")
    stream = torch.cuda.Stream()
    out = []
    with torch.cuda.stream(stream):
        call()
        stream.synchronize()
        h = ctypes.c_void_p(stream.cuda_stream)
        _ok(cu.cuStreamBeginCapture_v2(h, 2), "cuStreamBeginCapture")
        graph = ctypes.c_void_p()
        try:
            call()
        finally:
            status = cu.cuStreamEndCapture(h, ctypes.byref(graph))
        _ok(status, "cuStreamEndCapture")
    n = ctypes.c_size_t(0)
    _ok(cu.cuGraphGetNodes(graph, None, ctypes.byref(n)), "cuGraphGetNodes")
    nodes = (ctypes.c_void_p * n.value)()
    _ok(cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)), "cuGraphGetNodes")
    for node in nodes:
        kind = ctypes.c_int(-1)
        _ok(cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)), "cuGraphNodeGetType")
        if kind.value != 0:                 # CU_GRAPH_NODE_TYPE_KERNEL
            continue
        p = _Params()
        _ok(cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)), "cuGraphKernelNodeGetParams")
        name = ctypes.c_char_p()
        if p.func:
            _ok(cu.cuFuncGetName(ctypes.byref(name), ctypes.c_void_p(p.func)), "cuFuncGetName")
        else:
            _ok(cu.cuKernelGetName(ctypes.byref(name), ctypes.c_void_p(p.kern)), "cuKernelGetName")
        cluster = (ctypes.c_uint * 16)()
        # CU_LAUNCH_ATTRIBUTE_CLUSTER_DIMENSION
        _ok(cu.cuGraphKernelNodeGetAttribute(ctypes.c_void_p(node), 4, cluster), "cuGraphKernelNodeGetAttribute")
        out.append(_demangle(name.value.decode()) + (tuple(p.grid), tuple(p.block), max(1, cluster[0])))
    _ok(cu.cuGraphDestroy(graph), "cuGraphDestroy")
    return out
