"""Graph sweeps on both sides of the rule for staying on chip, against the oracle.

And that calls of small graphs with few classes take a launch per class where that
is faster: the kernels of a captured call.
"""
import numpy as np
import pytest

import oracle as O
import paper_1710_05155_gb300 as K
from test_gpu_planes_per_launch import _kernels

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,z,R,n,on_chip", [
    (64, 1, 64, 1, False), (64, 1, 128, 3, False), (64, 1, 64, 20, True), (10000, 2, 64, 20, False),
    (1000, 2, 64, 1, False), (1000, 2, 64, 20, True), (4096, 4, 64, 2, False), (4096, 4, 64, 10, True),
    (100, 4, 64, 1, True), (11000, 4, 64, 20, True)])
def test_choice_and_result(N, z, R, n, on_chip):
    import torch

    topo, m, stream = O.rrg(N, z, 3), min(2, z - 1), torch.cuda.Stream()
    with K.Simulation(topo=K.KA_RRG, N=N, z=z, m=m, replicas=R, graph_seed=3, stream=stream) as sim:
        sim.init(5, 0.6)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(graph, stream=stream):
            sim.sweep(n)
        assert (_kernels(graph) == 1) == (on_chip or n * sim.info["nclass"] == 1)
        graph.instantiate()
        graph.replay()
        torch.cuda.synchronize()
        st = O.init(N, R, 5, 0.6)
        O.sweeps(topo, m, st, 5, n)
        state, _, p = sim.get_state()
        assert np.array_equal(state, O.pack_words(st.n)) and np.array_equal(p, O.pack_words(st.p))
