"""The kernels a call launches, by name: the call is captured on its stream, so nothing runs, and the
graph is printed. The handle it is made on has counted steps that were never taken, and is
thrown away."""
import ctypes
import os
import re
import tempfile


def _cudart():
    with open("/proc/self/maps") as fh:
        paths = {line.split()[-1] for line in fh if "libcudart.so" in line}
    return ctypes.CDLL(sorted(paths)[0])  # the one torch has loaded


def launched(stream, call):
    """Mangled names, in launch order, of the kernels that call() queues on the torch stream."""
    rt, st = _cudart(), ctypes.c_void_p(stream.cuda_stream)
    graph = ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(st, 1) == 0  # thread-local
    try:
        call()
    finally:
        rc = rt.cudaStreamEndCapture(st, ctypes.byref(graph))
    assert rc == 0, rc
    fd, path = tempfile.mkstemp(suffix=".dot")
    os.close(fd)
    try:
        assert rt.cudaGraphDebugDotPrint(graph, path.encode(), 0) == 0
        with open(path) as fh:
            return re.findall(r'label="\d+\s*(_Z\w+)', fh.read())
    finally:
        os.unlink(path)
        rt.cudaGraphDestroy(graph)
