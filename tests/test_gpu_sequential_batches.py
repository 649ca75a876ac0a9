"""Random-sequential sweeps at the edges of the batches of 32 attempts and of the turns
of seven batches, against the oracle: sizes that are no multiple of 32, fewer batches than
makers, the largest planes kept in shared memory (stamps in what is left) and the first
beyond it, every z that shares the general instance.  Integer work: equality."""
import numpy as np
import pytest

import oracle as O
import paper_1710_05155_gb300 as K

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw,topo,sweeps", [
    (dict(topo=K.KA_RRG, N=6, z=3, m=1, replicas=64, graph_seed=1), lambda: O.rrg(6, 3, 1), 20),
    (dict(topo=K.KA_RRG, N=33, z=4, m=2, replicas=128, graph_seed=1), lambda: O.rrg(33, 4, 1), 9),
    (dict(topo=K.KA_RRG, N=250, z=5, m=2, replicas=64, graph_seed=1), lambda: O.rrg(250, 5, 1), 5),
    (dict(topo=K.KA_RRG, N=225, z=2, m=0, replicas=64, graph_seed=1), lambda: O.rrg(225, 2, 1), 5),
    (dict(topo=K.KA_CUBIC, d=2, L=100, m=1, replicas=64), lambda: O.cubic(2, 100), 2),
    (dict(topo=K.KA_CUBIC, d=2, L=104, m=1, replicas=256), lambda: O.cubic(2, 104), 1),
    (dict(topo=K.KA_CUBIC, d=3, L=20, m=5, replicas=64), lambda: O.cubic(3, 20), 2),
])
def test_batches(kw, topo, sweeps):
    t = topo()
    with K.Simulation(**kw) as sim:
        sim.init(17, 0.6)
        sim.sweep_sequential(sweeps)
        st = O.init(t.N, kw["replicas"], 17, 0.6)
        O.sequential_sweeps(t, kw["m"], st, 17, sweeps)
        n, _, p = sim.get_state()
        assert np.array_equal(n, O.pack_words(st.n)) and np.array_equal(p, O.pack_words(st.p))
