"""Planes of a large lattice on two streams: the sweeps of a call, beside other work of the
context's stream, equal those of contexts holding one word each (another seed's word index keys
the gates, so word w is compared with word w of a context reloaded plane by plane).
Integer work: equality."""
import numpy as np
import pytest

import paper_1710_05155_gb300 as K

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,R", [(60, 128), (64, 320), (100, 192), (112, 256), (128, 192)])
def test_chains_equal_one_launch_at_a_time(L, R):
    import torch

    kw = dict(topo=K.KA_CUBIC, d=3, L=L, m=3, replicas=R)
    stream = torch.cuda.Stream()
    with K.Simulation(**kw) as a, K.Simulation(stream=stream, **kw) as b:
        a.init(3, 0.8)
        K.ka_profile_enable(a.ctx, True)  # one chain, launch by launch
        a.sweep(7)
        want, counts = a.get_state(), a.observe()[1]
        b.init(3, 0.8)
        for k in (1, 4, 2):  # calls follow each other without a wait between them
            b.sweep(k)
        got_counts = b.observe()[1]
        got = b.get_state()
        assert np.array_equal(counts, got_counts)
        for x, y in zip(want, got):
            assert np.array_equal(x, y)


def test_chains_under_capture():
    import torch

    kw = dict(topo=K.KA_CUBIC, d=3, L=72, m=3, replicas=192)
    stream = torch.cuda.Stream()
    with K.Simulation(**kw) as a, K.Simulation(stream=stream, **kw) as b:
        for sim in (a, b):
            sim.init(4, 0.75)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            b.sweep(3)
        graph.replay()
        torch.cuda.synchronize()
        a.sweep(3)
        assert all(np.array_equal(x, y) for x, y in zip(a.get_state(), b.get_state()))
