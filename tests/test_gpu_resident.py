"""Small topologies whose sweeps stay on chip, against the oracle, word for word.

Shapes at the edges of the rules: the smallest and largest lattice and graph
of each cluster size, sides whose pencils do not divide evenly over the CTAs,
rows that leave lanes idle, graphs with missing neighbour slots (z < 4) and
with 32-byte records (z > 4), sites without room for the swapped bits, one
word and several, several sweeps per call.  Integer work: equality.
"""
import numpy as np
import pytest

import oracle as O
import paper_1710_05155_gb300 as K

pytestmark = pytest.mark.gpu


def _same(params, topo, seed, rho, steps):
    with K.Simulation(**params) as sim:
        sim.init(seed, rho)
        st = O.init(topo.N, params["replicas"], seed, rho)
        for k in steps:
            sim.sweep(k)
            O.sweeps(topo, params["m"], st, seed, k)
            n, n0, p = sim.get_state()
            assert np.array_equal(n, O.pack_words(st.n)), (params, st.t)
            assert np.array_equal(p, O.pack_words(st.p)), (params, st.t)
            assert np.array_equal(n0, O.pack_words(st.n0))


@pytest.mark.parametrize("d,L,R,m", [
    (2, 4, 64, 1), (2, 12, 192, 0), (2, 36, 128, 3), (2, 64, 64, 1), (2, 68, 64, 2),
    (2, 128, 128, 1), (3, 4, 64, 3), (3, 8, 320, 0), (3, 12, 192, 5), (3, 16, 64, 3),
    (3, 20, 64, 2), (3, 24, 320, 4), (3, 28, 320, 3), (4, 4, 64, 7), (4, 8, 128, 4),
    (4, 12, 256, 3), (3, 16, 64 * 160, 3),
])
def test_lattices(d, L, R, m):
    _same(dict(topo=K.KA_CUBIC, d=d, L=L, m=m, replicas=R), O.cubic(d, L), 11, 0.65,
          (1, 12) if L ** d * R < 1 << 20 else (3,))


@pytest.mark.parametrize("N,z,R,m", [
    (6, 3, 64, 1), (32, 1, 64, 0), (50, 5, 128, 3), (1001, 4, 192, 3), (1000, 2, 64, 0),
    (4096, 4, 64, 2), (8190, 4, 320, 2), (10998, 3, 64, 1), (11000, 4, 64 * 20, 2), (11001, 4, 64, 2),
    (16384, 4, 64, 2),
])
def test_random_regular_graphs(N, z, R, m):
    _same(dict(topo=K.KA_RRG, N=N, z=z, m=m, replicas=R, graph_seed=3), O.rrg(N, z, 3), 5, 0.6,
          (1, 5) if N * R < 1 << 20 else (4,))


@pytest.mark.parametrize("z,m", [(8, 0), (8, 5), (8, 7), (7, 3)])
def test_wide_neighbour_rows(z, m):
    N = 600
    steps = [k for k in range(1, z // 2 + 1)]
    nbr = np.array([sorted([(i + k) % N for k in steps] + [(i - k) % N for k in steps] +
                           ([(i + N // 2) % N] if z % 2 else [])) for i in range(N)], np.int32)
    _same(dict(topo=K.KA_GRAPH, N=N, z=z, m=m, replicas=128, nbr=nbr), O.graph(N, z, nbr.reshape(-1)),
          9, 0.6, (1, 5))


def test_batches_of_small_jobs():
    """One launch per shape class runs whole rounds: jobs of several sizes, words and targets."""
    jobs = [(dict(topo=K.KA_CUBIC, d=3, L=16, m=3, replicas=64), O.cubic(3, 16), 7),
            (dict(topo=K.KA_CUBIC, d=3, L=16, m=3, replicas=192), O.cubic(3, 16), 5),
            (dict(topo=K.KA_CUBIC, d=2, L=20, m=1, replicas=64), O.cubic(2, 20), 9),
            (dict(topo=K.KA_RRG, N=2000, z=4, m=2, replicas=256, graph_seed=2), O.rrg(2000, 4, 2), 6),
            (dict(topo=K.KA_RRG, N=3001, z=4, m=2, replicas=64, graph_seed=4), O.rrg(3001, 4, 4), 11),
            (dict(topo=K.KA_RRG, N=2000, z=3, m=2, replicas=64, graph_seed=5), O.rrg(2000, 3, 5), 8)]
    for flags in (K.KA_BATCH_GRAPH, 0):
        with K.Batch(flags=flags) as b:
            ids = [b.add(sweeps, 4, 21 + i, 0.7, **p) for i, (p, _, sweeps) in enumerate(jobs)]
            while b.step(3):
                pass
            for i, (p, topo, sweeps) in enumerate(jobs):
                st = O.init(topo.N, p["replicas"], 21 + i, 0.7)
                O.sweeps(topo, p["m"], st, 21 + i, sweeps)
                n, n0, pp = b.state(ids[i], p["replicas"] // 64, topo.N)
                assert np.array_equal(n, O.pack_words(st.n)), p
                assert np.array_equal(pp, O.pack_words(st.p)), p
                t, counts = b.observations(ids[i], p["replicas"])
                assert t[-1] == sweeps and np.array_equal(counts[-1], O.observe(st))


def test_last_sweep_number():
    """The sweep counter's last value: the resident kernels count sweeps, not end marks."""
    topo = O.cubic(3, 8)
    with K.Simulation(topo=K.KA_CUBIC, d=3, L=8, m=3, replicas=64) as sim:
        sim.init(3, 0.6)
        n, n0, p = sim.get_state()
        sim.set_state(n, n0, p, (1 << 32) - 9, 3)
        sim.sweep(9)
        st = O.init(topo.N, 64, 3, 0.6)
        st.t = (1 << 32) - 9
        O.sweeps(topo, 3, st, 3, 9)
        assert np.array_equal(sim.get_state()[0], O.pack_words(st.n))


@pytest.mark.parametrize("N,z,R", [(10999, 4, 64), (10999, 4, 256), (8190, 4, 320), (1000, 5, 128)])
def test_long_runs_equal_class_launches(N, z, R):
    """Classes of fewer bonds than CTAs: no CTA may run ahead of one without a bond.

    300 sweeps on chip, in a batch beside other jobs, against the same sweeps with a launch
    per class (as profiling runs them)."""
    kw = dict(topo=K.KA_RRG, N=N, z=z, m=2, replicas=R, graph_seed=7)
    with K.Simulation(**kw) as sim:
        sim.init(3, 0.7)
        K.ka_profile_enable(sim.ctx, True)
        sim.sweep(300)
        n, _, p = sim.get_state()
        K.ka_profile_enable(sim.ctx, False)
    with K.Batch() as b:
        ids = [b.add(300, 100, 3, 0.7, **kw) for _ in range(3)]
        b.add(300, 100, 5, 0.7, topo=K.KA_CUBIC, d=3, L=32, m=3, replicas=256)
        while b.step(25):
            pass
        for job in ids:
            bn, _, bp = b.state(job, R // 64, N)
            assert np.array_equal(bn, n) and np.array_equal(bp, p)
