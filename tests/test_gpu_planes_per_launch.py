"""ka_info's planes per launch against the kernel launches of captured sweeps."""
import ctypes as C

import pytest

import paper_1710_05155_gb300 as K

pytestmark = pytest.mark.gpu


def _kernels(graph) -> int:
    cuda = C.CDLL("libcuda.so.1")
    handle, count = C.c_void_p(graph.raw_cuda_graph()), C.c_size_t(0)
    assert cuda.cuGraphGetNodes(handle, None, C.byref(count)) == 0
    nodes = (C.c_void_p * count.value)()
    assert cuda.cuGraphGetNodes(handle, nodes, C.byref(count)) == 0
    kernels = 0
    for node in nodes:
        kind = C.c_int(-1)
        assert cuda.cuGraphNodeGetType(C.c_void_p(node), C.byref(kind)) == 0
        kernels += kind.value == 0  # CU_GRAPH_NODE_TYPE_KERNEL
    return kernels


# one chain of planes and two, all planes at once in two and a plane at a time; a
# square lattice's planes one by one; graphs with all planes in a launch
@pytest.mark.parametrize("params", [
    dict(topo=K.KA_CUBIC, d=3, L=L, m=3, replicas=R)
    for L, R in ((32, 128), (48, 256), (60, 128), (64, 64), (100, 192), (112, 320), (128, 256))
] + [dict(topo=K.KA_CUBIC, d=1, L=128, m=1, replicas=512)] + [
    dict(topo=K.KA_RRG, N=20000, z=4, m=2, replicas=R, graph_seed=1) for R in (64, 192, 512)
] + [dict(topo=K.KA_RRG, N=1 << 20, z=4, m=2, replicas=512, graph_seed=1)], ids=lambda p: f"{p.get('L', p.get('N'))}-{p['replicas']}")
def test_planes_per_launch_are_those_launched(params):
    import torch

    stream = torch.cuda.Stream()
    with K.Simulation(stream=stream, **params) as sim:
        sim.init(1, 0.7)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(graph, stream=stream):
            sim.sweep(2)  # a single sweep of a small lattice may take one chain of planes
        info = sim.info
        groups = info["nclass"] // 4 if params["topo"] == K.KA_CUBIC else info["nclass"]
        assert _kernels(graph) == 2 * groups * -(-info["planes"] // info["planes_per_launch"])
