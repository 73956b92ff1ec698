"""Stream capture through the CUDA runtime that torch has loaded, for tests of calls inside a caller's own capture."""
import ctypes

RELAXED = 2


def runtime():
    with open("/proc/self/maps") as f:
        path = next(l.split()[-1] for l in f if "libcudart.so" in l)
    lib = ctypes.CDLL(path)
    for name in ("cudaStreamBeginCapture", "cudaStreamEndCapture", "cudaGraphInstantiate", "cudaGraphLaunch",
                 "cudaGraphExecDestroy", "cudaGraphDestroy"):
        getattr(lib, name).restype = ctypes.c_int
    return lib


class Captured:
    """What `work()` enqueues on a stream (its handle), as a graph to replay; `status` is that of the capture's end."""

    def __init__(self, stream, work):
        self.lib, self.stream, self.exec = runtime(), ctypes.c_void_p(stream), ctypes.c_void_p()
        graph = ctypes.c_void_p()
        assert self.lib.cudaStreamBeginCapture(self.stream, RELAXED) == 0
        try:
            work()
        finally:
            self.status = self.lib.cudaStreamEndCapture(self.stream, ctypes.byref(graph))
            self.lib.cudaGetLastError()
        if self.status == 0:
            assert self.lib.cudaGraphInstantiate(ctypes.byref(self.exec), graph, ctypes.c_ulonglong(0)) == 0
            self.lib.cudaGraphDestroy(graph)

    def replay(self):
        assert self.lib.cudaGraphLaunch(self.exec, self.stream) == 0

    def close(self):
        if self.exec:
            self.lib.cudaGraphExecDestroy(self.exec)
            self.exec = None
