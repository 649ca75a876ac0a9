"""Group kernels at the sides where the pencil blocks cross layers and chunks are uneven: one
and several planes (the two forms of a side), every word against the oracle, two sweeps.
Integer work: equality."""
import numpy as np
import pytest

import oracle as O
import paper_1710_05155_gb300 as K

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,R,m", [(4, 64, 3), (12, 64, 2), (24, 64, 3), (36, 64, 1), (44, 64, 3),
                                   (60, 64, 3), (60, 128, 2), (64, 64, 4), (68, 64, 3), (68, 128, 3),
                                   (76, 64, 2), (100, 64, 3)])
def test_words_after_two_sweeps(L, R, m):
    with K.Simulation(topo=K.KA_CUBIC, d=3, L=L, m=m, replicas=R) as sim:
        sim.init(5, 0.7)
        K.ka_profile_enable(sim.ctx, True)  # a launch per group, also where sweeps stay on chip
        sim.sweep(2)
        n, _, p = sim.get_state()
    topo = O.cubic(3, L)
    for w in {0, R // 64 - 1}:
        st = O.init(L ** 3, 64, 5, 0.7, r0=64 * w)
        O.sweeps(topo, m, st, 5, 2)
        assert np.array_equal(n[w], O.pack_words(st.n)[0]), w
        assert np.array_equal(p[w], O.pack_words(st.p)[0]), w
