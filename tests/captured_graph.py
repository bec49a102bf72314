"""What a call enqueues on a stream, without running it: the call is captured
into a CUDA graph, and the graph's kernels and dependencies are read."""
import ctypes

PROGRAMMATIC = 1  # CU_GRAPH_DEPENDENCY_TYPE_PROGRAMMATIC


class _KernelParams(ctypes.Structure):
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("smem", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


class _EdgeData(ctypes.Structure):
    _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte),
                ("reserved", ctypes.c_ubyte * 5)]


def _ck(st):
    assert st == 0, f"CUDA driver error {st}"


def _kernel_name(cu, node):
    kind = ctypes.c_int()
    _ck(cu.cuGraphNodeGetType(node, ctypes.byref(kind)))
    if kind.value != 0:  # CU_GRAPH_NODE_TYPE_KERNEL
        return None
    p, name = _KernelParams(), ctypes.c_char_p()
    _ck(cu.cuGraphKernelNodeGetParams_v2(node, ctypes.byref(p)))
    if p.func:
        _ck(cu.cuFuncGetName(ctypes.byref(name), ctypes.c_void_p(p.func)))
    else:
        _ck(cu.cuKernelGetName(ctypes.byref(name), ctypes.c_void_p(p.kern)))
    return name.value.decode()


def captured(stream, call):
    """(kernel names, edges): the (mangled) names in the graph's node order, and
    per dependency (from name, to name, programmatic)."""
    cu = ctypes.CDLL("libcuda.so.1")
    vp = ctypes.c_void_p
    graph = vp()
    _ck(cu.cuStreamBeginCapture_v2(vp(stream), 1))  # thread-local
    try:
        call()
    finally:
        st = cu.cuStreamEndCapture(vp(stream), ctypes.byref(graph))
    _ck(st)
    try:
        n = ctypes.c_size_t()
        _ck(cu.cuGraphGetNodes(graph, None, ctypes.byref(n)))
        nodes = (vp * n.value)()
        _ck(cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)))
        names = {v: _kernel_name(cu, vp(v)) for v in nodes}
        m = ctypes.c_size_t()
        _ck(cu.cuGraphGetEdges_v2(graph, None, None, None, ctypes.byref(m)))
        a, b, d = (vp * m.value)(), (vp * m.value)(), (_EdgeData * m.value)()
        if m.value:
            _ck(cu.cuGraphGetEdges_v2(graph, a, b, d, ctypes.byref(m)))
        edges = [(names[a[k]], names[b[k]], d[k].type == PROGRAMMATIC) for k in range(m.value)]
        return [v for v in names.values() if v], edges
    finally:
        _ck(cu.cuGraphDestroy(graph))
