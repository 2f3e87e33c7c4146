"""What a captured graph is made of, read through the driver's graph calls."""
import ctypes

import torch

_KERNEL_NODE = 0
_PRIORITY = 8                      # CU_LAUNCH_ATTRIBUTE_PRIORITY


def _ok(status):
    assert status == 0, f"driver call failed with {status}"


def graph_roots(graph: torch.cuda.CUDAGraph) -> int:
    """Nodes without a predecessor: the branches that a capture begins with."""
    n = ctypes.c_size_t()
    _ok(ctypes.CDLL("libcuda.so.1").cuGraphGetRootNodes(ctypes.c_void_p(graph.raw_cuda_graph()), None, ctypes.byref(n)))
    return n.value


def kernel_priorities(graph: torch.cuda.CUDAGraph) -> list:
    """The launch priority of every kernel node."""
    cu = ctypes.CDLL("libcuda.so.1")
    g, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t()
    _ok(cu.cuGraphGetNodes(g, None, ctypes.byref(n)))
    nodes = (ctypes.c_void_p * n.value)()
    _ok(cu.cuGraphGetNodes(g, nodes, ctypes.byref(n)))
    out = []
    for node in nodes:
        kind = ctypes.c_int()
        _ok(cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)))
        if kind.value == _KERNEL_NODE:
            value = (ctypes.c_int * 16)()          # CUlaunchAttributeValue: 64 bytes
            _ok(cu.cuGraphKernelNodeGetAttribute(ctypes.c_void_p(node), _PRIORITY, value))
            out.append(value[0])
    return out
