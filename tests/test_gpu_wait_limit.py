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
    least = 1e9
    for k in range(5):  # the first call also loads the kernel
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
        end.synchronize()
        least = min(least, begin.elapsed_time(end))
    # 10 ms at least if it ran through
    assert least < 2.0, least
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


BATCH = """
import numpy as np, paper_1710_05155_gb300 as K
from paper_1710_05155_gb300 import serve, workloads
SMALL = [dict(topo=0, d=3, L=16, m=3, replicas=64), dict(topo=1, N=1000, z=4, m=2, replicas=64, graph_seed=1),
         dict(topo=1, N=8000, z=4, m=2, replicas=64, graph_seed=1)]
LARGE = dict(topo=0, d=3, L=32, m=3, replicas=128)  # no waits in its kernels
def refused(call, *args):
    try:
        call(*args)
    except K.KaError as e:
        return e.status == K.KA_ETIMEOUT
    return False
with K.Simulation(**LARGE) as sim:
    sim.init(3, 0.7)
    sim.sweep(40)
    want, counts = sim.get_state(), sim.observe()[1]
for flags in (K.KA_BATCH_GRAPH, 0, K.KA_BATCH_PLAIN):
    with K.Batch(flags=flags) as b:
        large = b.add(40, 20, 3, 0.7, **LARGE)
        b.step(10)
        small = [b.add(100, 50, 5, 0.7, **p) for p in SMALL]
        assert refused(b.step, 10)
        for job in small:
            assert b.poll(job)[1] and refused(b.observations, job, 64) and refused(b.state, job, 1, 1 << 14)
        assert b.info()["active"] == 1
        while b.info()["active"]:
            assert b.step(10)
        assert all(np.array_equal(x, y) for x, y in zip(b.state(large, 2, 32 ** 3), want))
        assert np.array_equal(b.observations(large, 128)[1][-1], counts)
        for job in small:
            b.remove(job)
        params, keep = K.make_params(**SMALL[0])
        ctx = K.ka_create(params, keep)
        K.ka_init(ctx, 3, 0.7)
        K.ka_sweep(ctx, 50)
        assert refused(b.adopt, ctx, 100, 50) and ctx
        K.ka_init(ctx, 3, 0.7)
        job = b.adopt(ctx, 100, 50)
        assert not refused(b.observations, job, 64) and refused(b.step, 20) and refused(b.state, job, 1, 4096)
jobs = [workloads.Job(p, 40, 20, 3, 0.7, 0.0, {}) for p in (LARGE, *SMALL)]
be = serve.DeviceBackend(0, 1 << 32, True, prepare_threads=2)
server = serve.Server(be, round_sweeps=10, autotune=False, keep_results=True)
report = server.run(jobs)
be.close()
assert report["done"] == 1 and report["failed"] == 3, report
assert [r.status for r in server.records] == ["done"] + 3 * ["failed"]
assert all("KA_ETIMEOUT" in r.error and r.counts is None for r in server.records[1:])
assert all(np.array_equal(x, y) for x, y in zip(server.records[0].state, want))
"""


def test_batches_and_served_jobs_say_so(library):
    variant.run(library, BATCH)
