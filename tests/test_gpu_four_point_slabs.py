"""Four-point sums where the padded lattice does not fit the scratch at once.

A chain of 33.6 million sites runs in slabs; a small lattice whose shells
reach half the side has vectors that are their own negative.  Against numpy's
shifted words.  Integer work: equality.
"""
import itertools

import numpy as np
import pytest

import paper_1710_05155_gb300 as K

pytestmark = pytest.mark.gpu


def _shells(q, d, L, smax, replicas):
    """phi of the given replicas, psi, from q words [R/64, N]."""
    W = q.shape[0]
    grid = q.reshape((W,) + (L,) * d)  # last axis = x
    M = np.bitwise_count(grid).sum(axis=0, dtype=np.int64)
    phi, psi = np.zeros((len(replicas), smax + 1), np.int64), np.zeros(smax + 1, np.int64)
    half = L // 2
    rad = int(np.sqrt(smax))
    for v in itertools.product(range(-min(rad, half), min(rad, half - 1) + 1), repeat=d):
        s = sum(c * c for c in v)
        if s > smax:
            continue
        shift, axes = tuple(-c for c in v), tuple(range(1, d + 1))
        both = grid & np.roll(grid, shift, axes)
        psi[s] += int((M * np.roll(M, shift, tuple(range(d)))).sum())
        for k, r in enumerate(replicas):
            phi[k, s] += int(((both[r // 64] >> np.uint64(r % 64)) & np.uint64(1)).sum())
    return phi, psi


@pytest.mark.parametrize("d,L,R,smax", [(1, 33_600_000, 64, 4), (2, 8, 128, 32), (3, 4, 64, 12),
                                        (3, 12, 64, 36), (2, 128, 64, 50)])
def test_padded_slabs(d, L, R, smax):
    with K.Simulation(topo=K.KA_CUBIC, d=d, L=L, m=1, replicas=R) as sim:
        sim.init(5, 0.6)
        sim.sweep(1)
        phi, psi = sim.four_point(smax)
        n, n0, _ = sim.get_state()
    replicas = (0, 37, R - 1)
    want, want_psi = _shells(n & n0, d, L, smax, replicas)
    assert np.array_equal(phi[list(replicas)], want)
    assert np.array_equal(psi, want_psi)
