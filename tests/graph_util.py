"""What a captured graph is made of, read through the driver's graph calls."""
import ctypes

import torch

_KERNEL_NODE = 0
_CLUSTER = 4                       # CU_LAUNCH_ATTRIBUTE_CLUSTER_DIMENSION
_PRIORITY = 8                      # CU_LAUNCH_ATTRIBUTE_PRIORITY


def _ok(status):
    assert status == 0, f"driver call failed with {status}"


def graph_roots(graph: torch.cuda.CUDAGraph) -> int:
    """Nodes without a predecessor: the branches that a capture begins with."""
    n = ctypes.c_size_t()
    _ok(ctypes.CDLL("libcuda.so.1").cuGraphGetRootNodes(ctypes.c_void_p(graph.raw_cuda_graph()), None, ctypes.byref(n)))
    return n.value


def _kernel_nodes(cu, graph: torch.cuda.CUDAGraph) -> list:
    g, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t()
    _ok(cu.cuGraphGetNodes(g, None, ctypes.byref(n)))
    nodes = (ctypes.c_void_p * n.value)()
    _ok(cu.cuGraphGetNodes(g, nodes, ctypes.byref(n)))
    out = []
    for node in nodes:
        kind = ctypes.c_int()
        _ok(cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)))
        if kind.value == _KERNEL_NODE:
            out.append(ctypes.c_void_p(node))
    return out


def _attribute(cu, node, which) -> list:
    value = (ctypes.c_int * 16)()          # CUlaunchAttributeValue: 64 bytes
    _ok(cu.cuGraphKernelNodeGetAttribute(node, which, value))
    return list(value)


def kernel_priorities(graph: torch.cuda.CUDAGraph) -> list:
    """The launch priority of every kernel node."""
    cu = ctypes.CDLL("libcuda.so.1")
    return [_attribute(cu, node, _PRIORITY)[0] for node in _kernel_nodes(cu, graph)]


class _KernelNodeParams(ctypes.Structure):          # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3), ("smem", ctypes.c_uint),
                ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p), ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def captured_kernels(call) -> list:
    """(mangled name, grid, block, CTAs of a cluster) of every kernel that `call` launches, read from a capture of it.  The
    call has run once before, so that nothing is set up under capture."""
    call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        call()
    cu = ctypes.CDLL("libcuda.so.1")
    out = []
    for node in _kernel_nodes(cu, graph):
        p, name = _KernelNodeParams(), ctypes.c_char_p()
        _ok(cu.cuGraphKernelNodeGetParams_v2(node, ctypes.byref(p)))
        if p.func:
            _ok(cu.cuFuncGetName(ctypes.byref(name), ctypes.c_void_p(p.func)))
        else:
            _ok(cu.cuKernelGetName(ctypes.byref(name), ctypes.c_void_p(p.kern)))
        out.append((name.value.decode(), tuple(p.grid), tuple(p.block), max(1, _attribute(cu, node, _CLUSTER)[0])))
    return out
