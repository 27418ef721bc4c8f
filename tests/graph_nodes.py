"""The kernels of a captured call and how they depend on one another, read back from the CUDA graph (nothing is launched)."""
import ctypes as C

import torch

_KERNEL_NODE, _PROGRAMMATIC = 0, 1


class _Edge(C.Structure):
    """CUgraphEdgeData"""
    _fields_ = [("from_port", C.c_ubyte), ("to_port", C.c_ubyte), ("type", C.c_ubyte), ("reserved", C.c_ubyte * 5)]


class _Params(C.Structure):
    """CUDA_KERNEL_NODE_PARAMS_v2"""
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("smem", C.c_uint),
                ("args", C.POINTER(C.c_void_p)), ("extra", C.POINTER(C.c_void_p)), ("kern", C.c_void_p), ("ctx", C.c_void_p)]


def _cu(name, *args):
    rc = getattr(C.CDLL("libcuda.so.1"), name)(*args)
    assert rc == 0, (name, rc)


class Captured:
    """The graph of what `call` enqueues on a side stream.  Calls that allocate scratch have to have run once before."""

    def __init__(self, call):
        self.g = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(self.g, capture_error_mode="thread_local"):
            call()
        h, n = C.c_void_p(self.g.raw_cuda_graph()), C.c_size_t()
        _cu("cuGraphGetNodes", h, None, C.byref(n))
        nodes = (C.c_void_p * n.value)()
        _cu("cuGraphGetNodes", h, nodes, C.byref(n))
        self.kernels = []                        # (name, parameters) in capture order
        for x in nodes:
            kind = C.c_int(-1)
            _cu("cuGraphNodeGetType", C.c_void_p(x), C.byref(kind))
            if kind.value == _KERNEL_NODE:
                p, name = _Params(), C.c_char_p()
                _cu("cuGraphKernelNodeGetParams_v2", C.c_void_p(x), C.byref(p))
                _cu("cuFuncGetName" if p.func else "cuKernelGetName", C.byref(name), C.c_void_p(p.func or p.kern))
                self.kernels.append((name.value.decode(), p))
        m = C.c_size_t()
        _cu("cuGraphGetEdges_v2", h, None, None, None, C.byref(m))
        src, dst, data = (C.c_void_p * m.value)(), (C.c_void_p * m.value)(), (_Edge * m.value)()
        if m.value:
            _cu("cuGraphGetEdges_v2", h, src, dst, data, C.byref(m))
        self.edge_types = [e.type for e in data]

    def programmatic(self):
        """How many kernels may start before the kernel in front of them has finished."""
        return self.edge_types.count(_PROGRAMMATIC)

    def argument(self, kernel, index, size):
        """Bytes of argument `index` of the captured kernel whose name holds `kernel`."""
        p = next(p for name, p in self.kernels if kernel in name)
        return C.string_at(p.args[index], size)
