"""Four-point sums of many words on a lattice whose staging plane holds few of them padded.

The sums of the first and last word against the oracle; and the time, which
passes word by word made 5.8 times that of an eighth of the words (a launch per
shell took 1.06 times): at most twice.
"""
import numpy as np
import pytest

import oracle as O
import paper_1710_05155_gb300 as K

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,L,R,smax", [(3, 8, 4096, 6), (2, 16, 4096, 25), (1, 128, 4096, 40), (3, 12, 256, 9)])
def test_first_and_last_word(d, L, R, smax):
    topo = O.cubic(d, L)
    with K.Simulation(topo=K.KA_CUBIC, d=d, L=L, m=2 * d - 1, replicas=R) as sim:
        sim.init(5, 0.7)
        sim.sweep(2)
        phi, _ = sim.four_point(smax)
    for w in (0, R // 64 - 1):
        st = O.init(topo.N, 64, 5, 0.7, r0=64 * w)
        O.sweeps(topo, 2 * d - 1, st, 5, 2)
        want, _ = O.four_point(d, L, st, smax)
        assert np.array_equal(phi[64 * w:64 * w + 64], want), w


def test_time():
    import time

    def least(R):
        with K.Simulation(topo=K.KA_CUBIC, d=3, L=8, m=3, replicas=R) as sim:
            sim.init(5, 0.7)
            times = []
            for _ in range(12):
                begin = time.perf_counter()
                sim.four_point(6)
                times.append(time.perf_counter() - begin)
            return min(times)

    assert least(4096) < 2 * least(512)
