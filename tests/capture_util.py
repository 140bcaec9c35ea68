"""The kernel launches a call enqueues, read off a stream capture of it (nothing runs on the GPU)."""
import ctypes
import os
import re
import tempfile

import torch


def launches(stream, call):
    """[(mangled kernel name, blocks, threads)] of what call() launches on `stream` (a torch.cuda.Stream)."""
    import pytest

    torch.cuda.current_device()
    try:
        rt = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    except OSError:
        pytest.skip("no shared CUDA runtime")
    handle, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(handle, 1) == 0  # thread-local mode
    try:
        call()
    finally:
        ended = rt.cudaStreamEndCapture(handle, ctypes.byref(graph))
    assert ended == 0
    with tempfile.TemporaryDirectory() as d:
        path = os.path.join(d, "graph.dot")
        assert rt.cudaGraphDebugDotPrint(graph, path.encode(), 4) == 0  # with kernel parameters
        text = open(path).read()
    rt.cudaGraphDestroy(graph)
    found = re.findall(r"(_Z\w+)\s*\\<\\<\\<(\{[\d, ]+\}|\d+), *(\{[\d, ]+\}|\d+),", text)
    count = lambda s: eval("*".join(re.findall(r"\d+", s)))  # noqa: E731
    return [(name, count(g), count(b)) for name, g, b in found]
