"""A job that is refused after its memory was taken leaves nothing behind."""
import numpy as np
import pytest

import paper_1710_05155_gb300 as K

pytestmark = pytest.mark.gpu


def test_a_refused_graph_is_harmless():
    rows = np.array([[(i + 1) % 64, (i - 1) % 64] for i in range(64)], np.int32)
    rows.sort(axis=1)
    wrong = rows.copy()
    wrong[5] = [7, 40]  # not symmetric
    with K.Batch() as b:
        with pytest.raises(K.KaError) as e:
            b.add(10, 5, 1, 0.7, topo=K.KA_GRAPH, N=64, z=2, m=1, replicas=64, nbr=wrong)
        assert e.value.status == K.KA_EINVAL
        assert b.info() == {"used_bytes": 0, "jobs": 0, "active": 0}
        job = b.add(10, 5, 1, 0.7, topo=K.KA_GRAPH, N=64, z=2, m=1, replicas=64, nbr=rows)
        while b.info()["active"]:
            b.step(5)
        assert b.poll(job) == (10, True)
