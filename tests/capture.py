"""Stream capture through the CUDA runtime's own calls (a capture that fails stays outside of torch)."""
import contextlib
import ctypes

import pytest

RELAXED = 2                                                  # cudaStreamCaptureModeRelaxed


def cudart():
    for name in ("libcudart.so.13", "/usr/local/cuda/lib64/libcudart.so"):
        try:
            return ctypes.CDLL(name)
        except OSError:
            pass
    pytest.skip("needs the CUDA runtime as a shared library")


@contextlib.contextmanager
def captured(stream):
    """What is enqueued on `stream` inside is captured and dropped."""
    rt, handle, graph = cudart(), ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(handle, RELAXED) == 0
    try:
        yield
    finally:
        rt.cudaStreamEndCapture(handle, ctypes.byref(graph))
        if graph.value:
            rt.cudaGraphDestroy(graph)
        rt.cudaGetLastError()
