"""On-chip sweeps whose waits run out.

In a test build every wait gives up at once.  The kernels must return, soon
and without a fault, and the calls must say that the state is not valid.
"""
import pytest

import variant

pytestmark = pytest.mark.gpu

UNITS = [f"ka_resident_cubic_d{d}" for d in (2, 3, 4)] + ["ka_resident_graph"]
# clusters of one, two, four and eight CTAs
PARAMS = [dict(topo=0, d=3, L=8, m=3, replicas=64), dict(topo=0, d=3, L=12, m=3, replicas=64),
          dict(topo=0, d=3, L=16, m=3, replicas=192), dict(topo=0, d=2, L=128, m=1, replicas=64),
          dict(topo=0, d=4, L=12, m=4, replicas=256),
          dict(topo=1, N=1000, z=4, m=2, replicas=64, graph_seed=1),
          dict(topo=1, N=8000, z=4, m=2, replicas=128, graph_seed=1)]


def _name(p):
    return f"d{p['d']}L{p['L']}" if "L" in p else f"N{p['N']}"


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    return variant.library(tmp_path_factory.mktemp("wait_limit"), UNITS, ["KA_WAIT_POLLS=0"])


LEAVES = """
import torch, paper_1710_05155_gb300 as K
with K.Simulation(**eval(sys.argv[1])) as sim:
    for k in range(2):  # the first call also loads the kernel
        sim.init(17, 0.6)
        begin, end = torch.cuda.Event(True), torch.cuda.Event(True)
        begin.record()
        sim.sweep(4096)
        end.record()
        try:
            sim.observe()
            raise SystemExit("no error")
        except K.KaError as e:
            assert e.status == K.KA_ETIMEOUT, e
    # 10 ms at least if it ran through
    assert begin.elapsed_time(end) < 2.0, begin.elapsed_time(end)
"""


@pytest.mark.parametrize("params", PARAMS, ids=_name)
def test_a_kernel_whose_wait_runs_out_leaves(library, params):
    variant.run(library, LEAVES, params)
