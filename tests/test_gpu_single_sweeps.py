"""Calls of one to three sweeps on both sides of the rules for staying on chip and for two
chains of planes: the launches of a captured call, and the state against one sweep at a
time while profiling (one launch after the other)."""
import numpy as np
import pytest

import paper_1710_05155_gb300 as K
from test_gpu_planes_per_launch import _kernels

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,R,n,kernels", [
    (12, 64, 1, 6), (12, 64, 2, 1), (16, 64, 3, 18), (16, 128, 2, 12), (16, 128, 3, 1), (64, 256, 1, 6),
    (64, 256, 2, 24), (80, 192, 1, 6), (80, 256, 1, 12), (80, 192, 3, 36)])
def test_launches_and_states(L, R, n, kernels):
    import torch

    kw, stream = dict(topo=K.KA_CUBIC, d=3, L=L, m=3, replicas=R), torch.cuda.Stream()
    with K.Simulation(stream=stream, **kw) as sim, K.Simulation(**kw) as other:
        sim.init(5, 0.7)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(graph, stream=stream):
            sim.sweep(n)
        assert _kernels(graph) == kernels
        graph.instantiate()
        graph.replay()
        torch.cuda.synchronize()
        other.init(5, 0.7)
        K.ka_profile_enable(other.ctx, True)
        for _ in range(n):
            other.sweep(1)
        assert all(np.array_equal(x, y) for x, y in zip(sim.get_state(), other.get_state()))
