"""Names of the kernels that a call launches, read from a capture of the
stream it launches on (nothing runs)."""
import ctypes


class _KernelParams(ctypes.Structure):  # CUDA_KERNEL_NODE_PARAMS of the driver API
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("shared", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def kernels(call, stream):
    """Kernel names (mangled) that call() launches on the torch stream."""
    cu = ctypes.CDLL("libcuda.so.1")

    def check(rc):
        assert rc == 0, rc

    st, graph, n = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    check(cu.cuStreamBeginCapture_v2(st, 1))   # thread-local mode
    try:
        call()
    finally:
        rc = cu.cuStreamEndCapture(st, ctypes.byref(graph))
    check(rc)
    check(cu.cuGraphGetNodes(graph, None, ctypes.byref(n)))
    nodes = (ctypes.c_void_p * n.value)()
    check(cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)))
    names = []
    for node in nodes:
        kind, p, name = ctypes.c_int(), _KernelParams(), ctypes.c_char_p()
        check(cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)))
        if kind.value != 0:
            continue
        check(cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)))
        if p.func:
            check(cu.cuFuncGetName(ctypes.byref(name), ctypes.c_void_p(p.func)))
        else:
            check(cu.cuKernelGetName(ctypes.byref(name), ctypes.c_void_p(p.kern)))
        names.append(name.value.decode())
    check(cu.cuGraphDestroy(graph))
    return names
