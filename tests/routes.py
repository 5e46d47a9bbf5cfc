"""Which kernels a call launches: the call is captured into a graph (nothing runs) and the graph's kernel nodes
are read through the driver."""
import ctypes as C
import re

import torch

NAME = re.compile(r"k_(?:leapfrog|adjoint|energy|res|wtb|rec|trace|init|flush)[a-z0-9_]*")


class _KernelParams(C.Structure):
    _fields_ = [("func", C.c_void_p), ("dims", C.c_uint * 7), ("params", C.c_void_p), ("extra", C.c_void_p),
                ("kern", C.c_void_p), ("ctx", C.c_void_p)]


def launches(call) -> list[str]:
    """Names (without template arguments) of the kernels that call(stream) enqueues, in order of their nodes."""
    cu = C.CDLL("libcuda.so.1")

    def ok(rc, what):
        assert rc == 0, (what, rc)

    s = torch.cuda.Stream()
    h = C.c_void_p(s.cuda_stream)
    graph = C.c_void_p()
    torch.cuda.synchronize()
    ok(cu.cuStreamBeginCapture_v2(h, 2), "begin")  # relaxed
    try:
        call(s)
    finally:
        rc = cu.cuStreamEndCapture(h, C.byref(graph))
    ok(rc, "end")
    n = C.c_size_t(0)
    ok(cu.cuGraphGetNodes(graph, None, C.byref(n)), "nodes")
    nodes = (C.c_void_p * n.value)()
    ok(cu.cuGraphGetNodes(graph, nodes, C.byref(n)), "nodes")
    out = []
    for node in nodes:
        kind = C.c_int()
        ok(cu.cuGraphNodeGetType(C.c_void_p(node), C.byref(kind)), "type")
        if kind.value != 0:  # a kernel
            continue
        p = _KernelParams()
        ok(cu.cuGraphKernelNodeGetParams_v2(C.c_void_p(node), C.byref(p)), "params")
        name = C.c_char_p()
        if p.func:
            ok(cu.cuFuncGetName(C.byref(name), C.c_void_p(p.func)), "name")
        else:
            ok(cu.cuKernelGetName(C.byref(name), C.c_void_p(p.kern)), "name")
        # the mangled name of the file, which ends in its own name, goes first
        out.append(NAME.findall(re.sub(r"_cu_[0-9a-f]{8}", " ", name.value.decode()))[-1])
    ok(cu.cuGraphDestroy(graph), "destroy")
    return out
