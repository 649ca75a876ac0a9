"""Initial states and counts at the edges of the one-pass selection, against the oracle.

Sizes on both sides of the list threshold (2048 sites), densities whose window
touches 0 or N, one particle and one hole, several words (also more than
sixteen, whose lists take turns), planes of 1, 2 and 4 words, breadth-first
graph order.  Integer work: equality.
"""
import numpy as np
import pytest

import oracle as O
import paper_1710_05155_gb300 as K

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw,topo", [
    (dict(topo=K.KA_CUBIC, d=1, L=32, m=1, replicas=64), lambda: O.cubic(1, 32)),
    (dict(topo=K.KA_CUBIC, d=3, L=12, m=3, replicas=192), lambda: O.cubic(3, 12)),
    (dict(topo=K.KA_CUBIC, d=2, L=44, m=1, replicas=64), lambda: O.cubic(2, 44)),
    (dict(topo=K.KA_CUBIC, d=2, L=48, m=1, replicas=1280), lambda: O.cubic(2, 48)),
    (dict(topo=K.KA_CUBIC, d=3, L=20, m=3, replicas=128), lambda: O.cubic(3, 20)),
    (dict(topo=K.KA_RRG, N=2047, z=4, m=2, replicas=64, graph_seed=3), lambda: O.rrg(2047, 4, 3)),
    (dict(topo=K.KA_RRG, N=2049, z=4, m=2, replicas=128, graph_seed=3), lambda: O.rrg(2049, 4, 3)),
    (dict(topo=K.KA_RRG, N=5000, z=3, m=1, replicas=1280, graph_seed=3), lambda: O.rrg(5000, 3, 3)),
])
def test_initial_states(kw, topo):
    t = topo()
    R = kw["replicas"]
    rhos = (0.85, 1.0 / t.N, 1.0 - 1.0 / t.N) if R > 1000 else \
        (0.0, 1.0, 0.5, 0.85, 1.0 / t.N, min(1.0, 40.0 / t.N), 1.0 - 1.0 / t.N)
    with K.Simulation(**kw) as sim:
        for k, rho in enumerate(rhos):
            sim.init(31 + k, rho)
            st = O.init(t.N, R, 31 + k, rho)
            n, n0, p = sim.get_state()
            assert np.array_equal(n, O.pack_words(st.n)), (kw, rho)
            assert np.array_equal(n0, n) and (p == np.uint64(2 ** 64 - 1)).all()
            assert np.array_equal(sim.observe()[1], O.observe(st))


@pytest.mark.parametrize("R,N", [(64, 1), (64, 2048 * 3 + 1), (128, 300_000), (4096, 130),
                                 (64, 800_001), (192, 500_001)])  # an odd number of fours a thread
def test_counts_of_arbitrary_planes(R, N):
    """Full, empty and random words: every digit of the counters, tails of every tile."""
    import torch

    g = np.random.default_rng(N)
    a = g.integers(0, 1 << 63, (3, R // 64, N), dtype=np.uint64) << np.uint64(1)
    a[0, 0] = np.uint64(2 ** 64 - 1)
    a[1, 0] = np.uint64(2 ** 64 - 1)
    t = torch.from_numpy(a.view(np.int64)).cuda()
    got = K.ka_observe_static(*(t[k].data_ptr() for k in range(3)), N, R,
                              torch.cuda.current_stream().cuda_stream)
    n, n0, p = a
    for o, x in enumerate((n, n & n0, n0 & p, p)):
        bits = np.unpackbits(x.view(np.uint8).reshape(R // 64, N, 8), axis=2, bitorder="little")
        assert np.array_equal(got[:, o], bits.sum(axis=1, dtype=np.int64).reshape(-1))
