"""The kernels of a call and the edges between them, from a stream capture (nothing runs)."""
import ctypes


class _KernelParams(ctypes.Structure):
    _fields_ = [("func", ctypes.c_void_p)] + [(k, ctypes.c_uint) for k in ("gx", "gy", "gz", "bx", "by", "bz", "smem")] + \
        [(k, ctypes.c_void_p) for k in ("params", "extra", "kern", "ctx")]


class _Edge(ctypes.Structure):
    _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte),
                ("reserved", ctypes.c_ubyte * 5)]


def _ok(rc):
    assert rc == 0, "driver call failed: %d" % rc


def captured(call):
    """call() under capture on a stream of its own: the kernels' mangled names in order of creation, and
    those (from, to) pairs of names whose edge is programmatic (an early start)."""
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    stream, graph, n = torch.cuda.Stream(), ctypes.c_void_p(), ctypes.c_size_t()
    st = ctypes.c_void_p(stream.cuda_stream)
    with torch.cuda.stream(stream):
        _ok(cu.cuStreamBeginCapture_v2(st, 2))  # relaxed
        try:
            call()
        finally:
            _ok(cu.cuStreamEndCapture(st, ctypes.byref(graph)))
    _ok(cu.cuGraphGetNodes(graph, None, ctypes.byref(n)))
    nodes = (ctypes.c_void_p * n.value)()
    _ok(cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)))
    names = {}
    for node in nodes:
        kind = ctypes.c_int()
        _ok(cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)))
        if kind.value:  # not a kernel
            continue
        p, name = _KernelParams(), ctypes.c_char_p()
        _ok(cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)))
        if p.func:
            _ok(cu.cuFuncGetName(ctypes.byref(name), ctypes.c_void_p(p.func)))
        else:
            _ok(cu.cuKernelGetName(ctypes.byref(name), ctypes.c_void_p(p.kern)))
        names[node] = name.value.decode()
    _ok(cu.cuGraphGetEdges_v2(graph, None, None, None, ctypes.byref(n)))
    a, b, e = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)(), (_Edge * n.value)()
    _ok(cu.cuGraphGetEdges_v2(graph, a, b, e, ctypes.byref(n)))
    early = [(names[a[i]], names[b[i]]) for i in range(n.value) if e[i].type == 1]
    _ok(cu.cuGraphDestroy(graph))
    return list(names.values()), early
