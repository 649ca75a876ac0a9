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


INVALID = """
import torch, numpy as np, paper_1710_05155_gb300 as K
def status(call, *args):
    try:
        call(*args)
        return K.KA_OK
    except K.KaError as e:
        return e.status
with K.Simulation(**eval(sys.argv[1])) as sim:
    sim.init(17, 0.6)
    state = sim.get_state()
    counts = torch.empty((sim.info["replicas"], 4), dtype=torch.int64, device="cuda")
    uses = [(sim.sweep, 1), (sim.observe,), (sim.get_state,), (sim.sweep_sequential, 1),
            (K.ka_observe_device, sim.ctx, counts.data_ptr())]
    if "L" in sys.argv[1]:
        uses.append((sim.four_point, 1))
    for valid in (lambda: sim.init(17, 0.6), lambda: sim.set_state(*state, 0, 17)):
        sim.sweep(50)
        assert status(K.ka_sync, sim.ctx) == K.KA_ETIMEOUT
        for u in uses:
            assert status(*u) == K.KA_ETIMEOUT, u
        valid()
        assert np.array_equal(sim.get_state()[0], state[0])
        assert sim.observe()[0] == 0
    if "L" in sys.argv[1]:
        sim.sweep(50)
        assert status(sim.four_point, 1) == K.KA_ETIMEOUT
"""


@pytest.mark.parametrize("params", [PARAMS[0], PARAMS[5]], ids=_name)
def test_the_state_stays_invalid_until_it_is_set_again(library, params):
    variant.run(library, INVALID, params)
