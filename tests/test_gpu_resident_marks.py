"""Swapped bits of on-chip lattice sweeps when some warps record theirs late.

A test build delays every second warp between reading and writing the record
of its swaps, so that the other warps are past the group's end meanwhile.
Every p plane must equal the oracle's.  Integer work: equality.
"""
import pytest

import variant

pytestmark = pytest.mark.gpu

CODE = """
import numpy as np, oracle as O, paper_1710_05155_gb300 as K
d, L, m, R = map(int, sys.argv[1:5])
topo = O.cubic(d, L)
with K.Simulation(topo=K.KA_CUBIC, d=d, L=L, m=m, replicas=R) as sim:
    sim.init(17, 0.6)
    st = O.init(topo.N, R, 17, 0.6)
    for k in (1, 2, 30):
        sim.sweep(k)
        O.sweeps(topo, m, st, 17, k)
        n, _, p = sim.get_state()
        assert np.array_equal(n, O.pack_words(st.n)) and np.array_equal(p, O.pack_words(st.p)), st.t
        assert np.array_equal(sim.observe()[1], O.observe(st))
"""


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    return variant.library(tmp_path_factory.mktemp("slow_marks"),
                           [f"ka_resident_cubic_d{d}" for d in (2, 3, 4)],
                           ["KA_SLOW_MARKS=if ((threadIdx.x >> 5) & 1) __nanosleep(3000)"])


# one CTA a word and clusters of two, four and eight; one word and several
@pytest.mark.parametrize("d,L,m,R", [(3, 8, 3, 64), (3, 12, 3, 64), (3, 16, 3, 192), (3, 20, 2, 64), (2, 32, 1, 64),
                                     (2, 64, 1, 128), (4, 8, 5, 64)])
def test_late_marks_are_kept(library, d, L, m, R):
    variant.run(library, CODE, d, L, m, R)
