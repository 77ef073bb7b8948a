"""Stream capture as a caller of the C library does it, through the CUDA
runtime that is loaded anyway."""
import ctypes

_rt = None
KERNEL = 0   # cudaGraphNodeTypeKernel


def _runtime():
    global _rt
    if _rt is None:
        _rt = ctypes.CDLL("libcudart.so.13")
    return _rt


def _ok(rc):
    assert rc == 0, f"cudaError {rc}"


class Captured:
    """The work that fn() puts on the stream (a torch stream), as a graph."""

    def __init__(self, stream, fn):
        rt = _runtime()
        self.stream = ctypes.c_void_p(stream.cuda_stream)
        self.graph = ctypes.c_void_p()
        _ok(rt.cudaStreamBeginCapture(self.stream, 1))   # thread-local
        try:
            fn()
        finally:
            rc = rt.cudaStreamEndCapture(self.stream, ctypes.byref(self.graph))
        _ok(rc)

    def kernels(self):
        """The number of kernel nodes."""
        rt = _runtime()
        n = ctypes.c_size_t()
        _ok(rt.cudaGraphGetNodes(self.graph, None, ctypes.byref(n)))
        nodes = (ctypes.c_void_p * n.value)()
        _ok(rt.cudaGraphGetNodes(self.graph, nodes, ctypes.byref(n)))
        kind = ctypes.c_int()
        count = 0
        for v in nodes:
            _ok(rt.cudaGraphNodeGetType(ctypes.c_void_p(v), ctypes.byref(kind)))
            count += kind.value == KERNEL
        return count

    def plain_edges(self):
        """Whether every edge is an ordinary one: asked without room for the
        edges' data, the query fails where an edge carries some."""
        rt = _runtime()
        n = ctypes.c_size_t()
        _ok(rt.cudaGraphGetEdges(self.graph, None, None, None, ctypes.byref(n)))
        if n.value == 0:
            return True
        a, b = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)()
        rc = rt.cudaGraphGetEdges(self.graph, a, b, None, ctypes.byref(n))
        assert rc in (0, 402), rc   # cudaErrorLossyQuery
        return rc == 0

    def replay(self, times=1):
        rt = _runtime()
        ex = ctypes.c_void_p()
        _ok(rt.cudaGraphInstantiate(ctypes.byref(ex), self.graph, ctypes.c_ulonglong(0)))
        for _ in range(times):
            _ok(rt.cudaGraphLaunch(ex, self.stream))
        _ok(rt.cudaStreamSynchronize(self.stream))
        _ok(rt.cudaGraphExecDestroy(ex))

    def close(self):
        _ok(_runtime().cudaGraphDestroy(self.graph))
