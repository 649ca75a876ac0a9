"""The work that a user has this library do, as cases that can be timed.

Each case goes through the public entry points (include/ka.h and its Python
binding): a simulation runs some sweeps, observes its replicas every few of
them and, at the end of the pass, hands its state over, in the canonical
layout, into page-locked host memory (what a program that keeps checkpoints
does).  The state goes on from pass to pass.  The sizes are those of the
repository's own configurations, benchmark, job mixes and tests.

Every output is a whole number (bit planes and counts), so there is nothing
for a calculation in 64-bit floating point to be compared with: ``exact``
gives ``None`` throughout.
"""
import torch

import paper_1710_05155_gb300 as K
from paper_1710_05155_gb300 import workloads

_LATTICE, _GRAPH = "lattice", "graph"


def listed():
    return [
        # the small configuration: one word per site, observed every 10 sweeps; the launches and the
        # wait for each observation count here
        {"name": "cubic_l16_r64", "kind": _LATTICE, "d": 3, "L": 16, "m": 3, "R": 64, "rho": 0.70,
         "sweeps": 100, "every": 10},
        # one replica word on a lattice whose rows are no power of two (request traces draw any
        # multiple of four)
        {"name": "cubic_l60_r64", "kind": _LATTICE, "d": 3, "L": 60, "m": 3, "R": 64, "rho": 0.80,
         "sweeps": 100, "every": 50},
        # a request of the served trace: three words per site, the other activation number
        {"name": "cubic_l100_r192", "kind": _LATTICE, "d": 3, "L": 100, "m": 2, "R": 192,
         "rho": 0.75, "sweeps": 50, "every": 50},
        # the benchmark's lattice, the largest side of the traces
        {"name": "cubic_l128_r256", "kind": _LATTICE, "d": 3, "L": 128, "m": 3, "R": 256,
         "rho": 0.85, "sweeps": 100, "every": 100},
        # the square lattice of the two-dimensional model
        {"name": "square_l128_r256", "kind": _LATTICE, "d": 2, "L": 128, "m": 1, "R": 256,
         "rho": 0.70, "sweeps": 100, "every": 50},
        # a small graph of the job mixes: one word per site, a class is a few hundred warps
        {"name": "rrg_n14_r64", "kind": _GRAPH, "N": 1 << 14, "z": 4, "m": 2, "R": 64, "rho": 0.80,
         "rho_last": 0.80, "sweeps": 100, "every": 50},
        # the density scan on the large random regular graph: eight densities as the eight words
        {"name": "rrg_n20_scan", "kind": _GRAPH, "N": 1 << 20, "z": 4, "m": 2, "R": 512,
         "rho": 0.55, "rho_last": 0.90, "sweeps": 30, "every": 30},
        # many independent jobs advanced together, from one observation to the next
        {"name": "batch_mix_26", "kind": "batch", "jobs": 26, "mix": 1, "every": 100, "round": 25},
        # the initial state of the benchmark's lattice (every run and every served job begins so)
        {"name": "init_l128_r256", "kind": "init", "L": 128, "R": 256, "rho": 0.85},
        # one observation of that lattice, left on the device
        {"name": "observe_l128_r256", "kind": "observe", "L": 128, "R": 256, "rho": 0.85},
        # space-dependent correlations out to r = 5
        {"name": "four_point_l64_r256", "kind": "four_point", "d": 3, "L": 64, "R": 256,
         "rho": 0.80, "smax": 25},
        # the random-sequential schedule of the original method
        {"name": "sequential_l16_r256", "kind": "sequential", "L": 16, "R": 256, "m": 3,
         "rho": 0.70, "sweeps": 20},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _replicas(rng, largest=256):
    return 64 * rng.randint(1, largest // 64)


def draw(rng):
    kind = rng.choice([_LATTICE] * 4 + [_GRAPH] * 3 +
                      ["square", "batch", "init", "observe", "four_point", "sequential"])
    rho = round(rng.uniform(0.55, 0.90), 3)
    if kind == _LATTICE:
        side, R, m = 4 * _log_int(rng, 4, 32), _replicas(rng), rng.choice([2, 3])
        every = rng.choice([5, 10, 20, 50])
        return {"kind": _LATTICE, "d": 3, "L": side, "m": m, "R": R,
                "rho": round(rng.uniform(0.70, 0.90), 3), "sweeps": every * rng.randint(1, 50 // every),
                "every": every}
    if kind == "square":
        d = rng.choice([2, 2, 4])
        side = 4 * (_log_int(rng, 4, 32) if d == 2 else rng.randint(2, 5))
        return {"kind": _LATTICE, "d": d, "L": side, "m": rng.choice([1, 2]) if d == 2 else 4,
                "R": _replicas(rng), "rho": rho, "sweeps": 40, "every": rng.choice([10, 20, 40])}
    if kind == _GRAPH:
        z, m = rng.choice([(4, 2), (4, 2), (4, 3), (3, 1)])
        n = 2 * _log_int(rng, 1 << 11, 1 << 19)
        R = _replicas(rng)
        return {"kind": _GRAPH, "N": n, "z": z, "m": m, "R": R, "rho": rho,
                "rho_last": rng.choice([rho, 0.9]), "sweeps": 40, "every": rng.choice([10, 40])}
    if kind == "batch":
        return {"kind": "batch", "jobs": rng.randint(8, 26), "mix": rng.randint(2, 10 ** 6),
                "every": 50, "round": rng.choice([10, 25, 50])}
    side, R = 4 * _log_int(rng, 4, 32), _replicas(rng)
    if kind in ("init", "observe"):
        return {"kind": kind, "L": side, "R": R, "rho": rho}
    if kind == "four_point":
        d = rng.choice([2, 3, 3])
        side = 4 * rng.randint(3, 16)
        return {"kind": kind, "d": d, "L": side, "R": R, "rho": rho, "smax": rng.randint(1, 25)}
    return {"kind": kind, "L": 4 * rng.randint(2, 5), "R": R, "m": rng.choice([2, 3]), "rho": rho,
            "sweeps": rng.randint(2, 10)}


class _Run:
    """A simulation and the page-locked host arrays that its state is handed over in."""

    def __init__(self, arrays, **params):
        self.sim = K.Simulation(**params)
        info = self.sim.info
        self.words, self.sites = info["words"], info["N"]
        self.host = {k: torch.empty((self.words, self.sites), dtype=torch.int64, pin_memory=True)
                     for k in arrays}

    def state(self):
        """The planes asked for, read into the host arrays (n0 never changes in a run)."""
        pointers = [self.host[k].data_ptr() if k in self.host else None for k in ("n", "n0", "p")]
        status = K.load().ka_get_state(self.sim.ctx.handle, *pointers)
        if status != K.KA_OK:
            raise K.KaError(status, "ka_get_state")
        return dict(self.host)


def _lattice(case, arrays=("n", "p"), **more):
    return _Run(arrays, topo=K.KA_CUBIC, d=case.get("d", 3), L=case["L"], m=case.get("m", 3),
                replicas=case["R"], **more)


def _seeded(seed, k=0):
    return (seed * 1000003 + k) % (1 << 62) + 1


def _densities(case):
    """One density per replica word, evenly spaced from rho to rho_last."""
    w = case["R"] // 64
    step = (case["rho_last"] - case["rho"]) / max(1, w - 1)
    return [case["rho"] + k * step for k in range(w)]


def _jobs(case):
    """The jobs of the repository's own instance mix (sides 16 to 96, graphs of 2^12 to 2^18 sites)."""
    return workloads.instance_mix(case["jobs"], case["mix"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == _LATTICE:
        r = _lattice(case)
        r.sim.init(_seeded(seed), case["rho"])
        return case, r
    if kind == _GRAPH:
        r = _Run(("n", "p"), topo=K.KA_RRG, N=case["N"], z=case["z"], m=case["m"],
                 replicas=case["R"], graph_seed=1)
        rhos = _densities(case)
        if len(set(rhos)) == 1:
            r.sim.init(_seeded(seed), rhos[0])
            return case, r
        words = []
        for w, rho in enumerate(rhos):
            r.sim.init(_seeded(seed, w), rho)
            words.append(r.state()["n"][w].clone())
        n = torch.stack(words).numpy().view("u8")
        r.sim.set_state(n, n, torch.full(n.shape, -1, dtype=torch.int64).numpy().view("u8"), 0,
                        _seeded(seed))
        return case, r
    if kind == "batch":
        batch = K.Batch()
        jobs = []
        for k, j in enumerate(_jobs(case)):
            job = batch.add(400_000, case["every"], _seeded(seed, k), j.rho,
                            **dict(j.params, **({"graph_seed": k + 1} if "N" in j.params else {})))
            jobs.append((job, j.params["replicas"] // 64 * j.sites))
        total = sum(n for _, n in jobs)
        host = {k: torch.empty(total, dtype=torch.int64, pin_memory=True) for k in ("n", "p")}
        return case, batch, jobs, host
    if kind == "init":
        return case, _lattice(case, ("n",)), _seeded(seed)
    if kind == "observe":
        r = _lattice(case, ())
        r.sim.init(_seeded(seed), case["rho"])
        r.sim.sweep(20)
        return case, r, torch.empty((case["R"], 4), dtype=torch.int64, device="cuda")
    if kind == "four_point":
        r = _lattice(case, ())
        r.sim.init(_seeded(seed), case["rho"])
        r.sim.sweep(20)
        return case, r
    r = _lattice(case)
    r.sim.init(_seeded(seed), case["rho"])
    return case, r


def _run_batch(case, batch, jobs, host):
    every, done = case["every"], 0
    while done < every:
        done += batch.step(min(case["round"], every - done))
    at = 0
    for job, n in jobs:
        status = K.load().ka_batch_state(batch.handle, job, host["n"][at:].data_ptr(), None,
                                         host["p"][at:].data_ptr())
        if status != K.KA_OK:
            raise K.KaError(status, "ka_batch_state")
        at += n
    return dict(host)


def run(state):
    case, r = state[:2]
    kind = case["kind"]
    if kind in (_LATTICE, _GRAPH):
        counts = []
        for _ in range(case["sweeps"] // case["every"]):
            r.sim.sweep(case["every"])
            counts.append(r.sim.observe()[1])
        return {"counts": counts, **r.state()}
    if kind == "batch":
        return _run_batch(*state)
    if kind == "init":
        r.sim.init(state[2], case["rho"])
        return r.state()
    if kind == "observe":
        K.ka_observe_device(r.sim.ctx, state[2].data_ptr())
        return state[2]
    if kind == "four_point":
        return r.sim.four_point(case["smax"])
    r.sim.sweep_sequential(case["sweeps"])
    return r.state()


# 32-bit integer operations of one Philox4x32-10 block: per round two wide multiplications and two
# three-input exclusive ors
_BLOCK = 40


def work(case):
    """Bytes: a sweep reads and writes n and p once (16 bytes a site-word), a graph's sweep reads its
    neighbour rows and bonds too, an observation reads n, n0 and p, and the state handed over is
    written once.  "flops": the 32-bit operations of the random blocks, which no sweep or initial
    state does without (half a block a bond and word; half a block a site and replica), and for
    four_point one AND and one addition (of a bit-sliced counter) per pair of words and vector."""
    kind = case["kind"]
    if kind == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for j in _jobs(case):
            z = j.params.get("z", 6)
            one = _sweeps(j.sites, z, j.params["replicas"] // 64, case["every"], 1, "N" in j.params)
            total = {k: total[k] + one[k] for k in total}
        return total
    sites = case["N"] if kind == _GRAPH else case["L"] ** case.get("d", 3)
    w = case["R"] // 64
    if kind in (_LATTICE, _GRAPH):
        z = case["z"] if kind == _GRAPH else 2 * case["d"]
        return _sweeps(sites, z, w, case["sweeps"], case["sweeps"] // case["every"], kind == _GRAPH)
    if kind == "init":
        return {"bytes": 32.0 * sites * w, "flops": 32.0 * _BLOCK * sites * w}
    if kind == "observe":
        return {"bytes": 24.0 * sites * w + 32.0 * case["R"], "flops": 0.0}
    if kind == "four_point":
        vectors = _vectors(case["d"], case["L"], case["smax"])
        return {"bytes": 16.0 * sites * w + 8.0 * (case["R"] + 1) * (case["smax"] + 1),
                "flops": 4.0 * sites * w * vectors / 2}
    return {"bytes": (32.0 * case["sweeps"] + 16.0) * sites * w,
            "flops": float(_BLOCK) * sites * w * case["sweeps"]}


def _sweeps(sites, z, w, sweeps, observations, graph):
    tables = sites * (4.0 * z + 6.0 * z) if graph else 0.0
    return {"bytes": sites * w * (32.0 * sweeps + 24.0 * observations + 16.0) + tables * sweeps,
            "flops": _BLOCK * sites * w * sweeps * z / 4.0}


def _vectors(d, side, smax):
    """Displacement vectors of length squared at most smax with components in [-side/2, side/2)."""
    counts = {0: 1}
    for _ in range(d):
        more = {}
        for s, n in counts.items():
            for x in range(-(side // 2), side // 2):
                if s + x * x <= smax:
                    more[s + x * x] = more.get(s + x * x, 0) + n
        counts = more
    return sum(counts.values())


def exact(case, seed):
    return None
