import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

GOLDEN = os.path.join(ROOT, "tests", "golden")


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (B200, sm_100a)")


def golden_lines(name):
    """Non-comment, non-empty lines of a golden text fixture."""
    with open(os.path.join(GOLDEN, name)) as f:
        return [ln.strip() for ln in f if ln.strip() and not ln.lstrip().startswith("#")]


def pair_launches(call):
    """How many of the kernels that `call` launches run as pairs of CTAs (clusters of two asked for at the launch), from a
    capture of the call; nothing is executed."""
    import ctypes
    import torch
    graph, stream = torch.cuda.CUDAGraph(keep_graph=True), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        graph.capture_begin()
        call()
        graph.capture_end()
    cuda = ctypes.CDLL("libcuda.so.1")
    handle, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert cuda.cuGraphGetNodes(handle, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cuda.cuGraphGetNodes(handle, nodes, ctypes.byref(n)) == 0
    pairs = 0
    for node in nodes:
        kind, dims = ctypes.c_int(), (ctypes.c_uint * 16)()                # CUlaunchAttributeValue: 64 bytes
        assert cuda.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value == 0:                                                # a kernel; attribute 4: its cluster's size
            assert cuda.cuGraphKernelNodeGetAttribute(ctypes.c_void_p(node), 4, dims) == 0
            pairs += tuple(dims[:3]) == (2, 1, 1)
    return pairs


@pytest.fixture(scope="session")
def lib():
    """The CUDA library through its Python binding; fails loudly if it is not built."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2501_17116_b200 as fp4
    return fp4
