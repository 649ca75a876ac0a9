"""Class launches of graphs too large for the on-chip kernels: planes of 1, 2 and 4 words,
planes run together and one after another, and in batches of uneven sizes, against the oracle
run on some replica words alone.  Integer work: equality."""
import numpy as np
import pytest

import oracle as O
import paper_1710_05155_gb300 as K

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,z,m,R", [(30001, 4, 2, 64), (30001, 4, 3, 128), (40002, 3, 1, 192),
                                     (30002, 4, 1, 512), (32000, 2, 0, 256)])
def test_words_of_planes(N, z, m, R):
    topo = O.rrg(N, z, 2)
    with K.Simulation(topo=K.KA_RRG, N=N, z=z, m=m, replicas=R, graph_seed=2) as sim:
        sim.init(9, 0.6)
        sim.sweep(2)
        n, _, p = sim.get_state()
    for w in {0, R // 64 - 1}:
        st = O.init(N, 64, 9, 0.6, r0=64 * w)
        O.sweeps(topo, m, st, 9, 2)
        assert np.array_equal(n[w], O.pack_words(st.n)[0]), w
        assert np.array_equal(p[w], O.pack_words(st.p)[0]), w


def test_batches_of_large_graphs():
    jobs = [(30000, 4, 2, 64), (50000, 4, 2, 64), (61001, 4, 2, 64), (130000, 4, 2, 64),
            (30000, 4, 2, 256), (40000, 3, 2, 128)]
    for flags in (K.KA_BATCH_GRAPH, 0):
        with K.Batch(flags=flags) as b:
            ids = [b.add(5 + i, 4, 40 + i, 0.75, topo=K.KA_RRG, N=N, z=z, m=m, replicas=R, graph_seed=2)
                   for i, (N, z, m, R) in enumerate(jobs)]
            while b.step(3):
                pass
            for i, (N, z, m, R) in enumerate(jobs):
                st = O.init(N, 64, 40 + i, 0.75)
                O.sweeps(O.rrg(N, z, 2), m, st, 40 + i, 5 + i)
                n, _, p = b.state(ids[i], R // 64, N)
                assert np.array_equal(n[0], O.pack_words(st.n)[0]) and np.array_equal(p[0], O.pack_words(st.p)[0])
