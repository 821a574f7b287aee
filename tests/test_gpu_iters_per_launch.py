"""CUPSO_OPT_ITERS_PER_LAUNCH: how many kernels a cupso_step call launches, counted in a captured graph."""
import ctypes

import pytest

from tests.gpu_common import load_cupso

pytestmark = pytest.mark.gpu

BOX = (-100.0, 100.0, 20.0)


def _kernels_of(graph):
    rt = ctypes.CDLL("libcudart.so.13")
    n = ctypes.c_size_t()
    g = ctypes.c_void_p(graph)
    assert rt.cudaGraphGetNodes(g, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(g, nodes, ctypes.byref(n)) == 0
    kinds = []
    for node in nodes:
        kind = ctypes.c_int()
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kinds.append(kind.value)
    return kinds.count(0)   # cudaGraphNodeTypeKernel


@pytest.mark.parametrize("dtype,mode,per_launch,launches", [
    ("f32", "sync", 0, 1), ("f32", "sync", 8, 3), ("f32", "sync", 1, 20),
    ("f64", "sync", 0, 1), ("f64", "sync", 8, 3), ("f64", "sync", 1, 20), ("f64", "persistent", 8, 1)])
def test_launches_of_a_call(dtype, mode, per_launch, launches):
    P = load_cupso()
    import torch

    stream = torch.cuda.Stream()
    with P.Swarm(7, 5000, BOX, 1.0, 2.0, 2.0, 0, 5, mode=mode, dtype=dtype, stream=stream.cuda_stream) as s:
        s.set_option(P.CUPSO_OPT_ITERS_PER_LAUNCH, per_launch)
        s.set_option(P.CUPSO_OPT_GRAPH_CHUNK, 0)
        graph = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(graph, stream=stream):
            s.step(20)
        assert _kernels_of(graph.raw_cuda_graph()) == launches
