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


def _launches(P, s, iters):
    import torch

    stream = torch.cuda.Stream()
    s.set_stream(stream.cuda_stream)
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph, stream=stream):
        s.step(iters)
    return _kernels_of(graph.raw_cuda_graph())


@pytest.mark.parametrize("dtype,mode,per_launch,launches", [
    ("f32", "sync", 0, 1), ("f32", "sync", 8, 3), ("f32", "sync", 1, 20),
    ("f64", "sync", 0, 1), ("f64", "sync", 8, 3), ("f64", "sync", 1, 20), ("f64", "persistent", 8, 1)])
def test_launches_of_a_call(dtype, mode, per_launch, launches):
    P = load_cupso()
    with P.Swarm(7, 5000, BOX, 1.0, 2.0, 2.0, 0, 5, mode=mode, dtype=dtype) as s:
        s.set_option(P.CUPSO_OPT_ITERS_PER_LAUNCH, per_launch)
        s.set_option(P.CUPSO_OPT_GRAPH_CHUNK, 0)
        assert _launches(P, s, 20) == launches


@pytest.mark.parametrize("dtype,mode,N,D", [("f32", "sync", 5000, 30), ("f32", "sync", 1, 1), ("f32", "auto", 1024, 32),
                                            ("f32", "sync", 1 << 18, 32), ("f32", "tree", 5000, 30),
                                            ("f64", "sync", 8192, 1), ("f64", "persistent", 500, 7),
                                            ("f64", "sync", 30000, 10), ("f64", "queue", 500, 7)])
def test_info_says_from_where_a_call_is_one_launch(dtype, mode, N, D):
    P = load_cupso()
    with P.Swarm(D, N, BOX, 1.0, 2.0, 2.0, 0, 5, mode=mode, dtype=dtype) as s:
        s.set_option(P.CUPSO_OPT_GRAPH_CHUNK, 0)
        n = s.info()["one_launch_iters"]
        assert (n > 0) == (mode in ("sync", "auto", "persistent") and N * D <= 1 << 20)
        if n:
            assert _launches(P, s, n) == 1
            assert mode != "sync" or _launches(P, s, n - 1) == n - 1
            s.set_option(P.CUPSO_OPT_ITERS_PER_LAUNCH, 1)
            assert s.info()["one_launch_iters"] == (1 if mode == "persistent" else 0)
