"""What a call launches: the kernel nodes of its work captured into a graph
(never run), read back through the CUDA driver API."""
import ctypes as C


class _KernelParams(C.Structure):
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("smem", C.c_uint),
                ("params", C.c_void_p), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]


_CLUSTER, _PRIORITY = 4, 8  # CUlaunchAttributeID


def kernel_launches(call, stream):
    """[(grid x, block x, cluster x, priority)] of the kernels `call()` puts on `stream` (a torch stream)."""
    cu = C.CDLL("libcuda.so.1")

    def ok(rc):
        assert rc == 0, rc

    st = C.c_void_p(stream.cuda_stream)
    graph = C.c_void_p()
    ok(cu.cuStreamBeginCapture_v2(st, C.c_int(1)))  # thread-local mode
    try:
        call()
    finally:
        rc = cu.cuStreamEndCapture(st, C.byref(graph))
    ok(rc)
    n = C.c_size_t(0)
    ok(cu.cuGraphGetNodes(graph, None, C.byref(n)))
    nodes = (C.c_void_p * n.value)()
    ok(cu.cuGraphGetNodes(graph, nodes, C.byref(n)))
    out = []
    for h in nodes:
        node, kind = C.c_void_p(h), C.c_int(-1)
        ok(cu.cuGraphNodeGetType(node, C.byref(kind)))
        if kind.value != 0:  # not a kernel
            continue
        p = _KernelParams()
        ok(cu.cuGraphKernelNodeGetParams_v2(node, C.byref(p)))
        val = []
        for attr in (_CLUSTER, _PRIORITY):
            v = (C.c_int * 16)()  # (the attribute union: 64 bytes)
            ok(cu.cuGraphKernelNodeGetAttribute(node, C.c_int(attr), v))
            val.append(v[0])
        out.append((p.grid[0], p.block[0], max(val[0], 1), val[1]))
    ok(cu.cuGraphDestroy(graph))
    return out
