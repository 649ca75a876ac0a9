"""Contexts of different sizes swept from two host threads at once.

Their launches share kernel instances but want different amounts of shared
memory.  Every launch must succeed, and the states equal those of the same
sweeps from one thread.
"""
import threading

import numpy as np
import pytest

import paper_1710_05155_gb300 as K

pytestmark = pytest.mark.gpu

CALLS = 2000
GRAPHS = [dict(topo=K.KA_RRG, N=N, z=4, m=2, replicas=64, graph_seed=3) for N in (6000, 10000)]
LATTICES = [dict(topo=K.KA_CUBIC, d=3, L=L, m=3, replicas=64) for L in (8, 20)]


@pytest.mark.parametrize("params,call,sweeps", [(GRAPHS, "sweep", 4), (LATTICES, "sweep_sequential", 1)],
                         ids=["graphs", "sequential"])
def test_two_threads(params, call, sweeps):
    import torch

    sims = [K.Simulation(stream=torch.cuda.Stream(), **p) for p in params]
    errors = []

    def run(sim):
        try:
            for _ in range(CALLS):
                getattr(sim, call)(sweeps)
        except K.KaError as e:
            errors.append(e)

    for sim in sims:
        sim.init(5, 0.7)
    threads = [threading.Thread(target=run, args=(s,)) for s in sims]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for sim, p in zip(sims, params):
        with K.Simulation(**p) as alone:
            alone.init(5, 0.7)
            for _ in range(CALLS):
                getattr(alone, call)(sweeps)
            for x, y in zip(sim.get_state(), alone.get_state()):
                assert np.array_equal(x, y)
        sim.close()
