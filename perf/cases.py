"""Performance cases of the solver: what its users run, through its public entry points.

A case is a plain dict: ``kind`` says which entry points it takes, the rest are
sizes and parameters. ``listed()`` gives the fixed cases, ``draw()`` more of the
same ranges, ``prepare()`` what a user's program holds before the call,
``run()`` one pass, ``work()`` the bytes and operations a pass cannot do
without, and ``exact()`` the outputs of a pass from plain 64-bit arithmetic.

Most outputs are whole numbers (cuts, bisectors, spins, energies). A trial is
a long switched dynamical system, so its outputs have no value that 64-bit
arithmetic could give independently of the rounding of every step; a readout
of given phases has one, and ``exact()`` gives it.
"""
import math

import numpy as np
import torch

import paper_2605_30355_gb300 as cosm

STORAGE = {"f32": cosm.F32, "f16": cosm.F16, "q16": cosm.Q16, "bf16": cosm.BF16}

# the largest listed case's edge-replica updates; a drawn case does no more
MOST_UPDATES = 40000 * 1024 * 2000


def listed():
    torus = dict(alpha0=14.0, ratio=0.5, period=3)
    graph = dict(alpha0=14.0, ratio=1.0, period=3)
    return [
        # the smallest call: a 256-spin lattice, 64 trials of 1,000 sweeps; launches and latency count
        dict(name="trial_torus16_f32", kind="trial", graph="torus2d", L1=16, L2=16, storage="f32",
             replicas=64, sweeps=1000, **torus),
        # the headline workload's shape (20,000-spin 2D glass, 1,024 trials) with a short anneal
        dict(name="trial_torus20k_f32", kind="trial", graph="torus2d", L1=100, L2=200, storage="f32",
             replicas=1024, sweeps=2000, **torus),
        # the same in the 2-byte form that keeps binary32's success rate
        dict(name="trial_torus20k_q16", kind="trial", graph="torus2d", L1=100, L2=200, storage="q16",
             replicas=1024, sweeps=2000, **torus),
        # one-shot call on host buffers: graph in, best spins and all cuts out, nothing kept
        dict(name="solve_torus10k_f16", kind="solve", graph="torus2d", L1=100, L2=100, storage="f16",
             replicas=1024, sweeps=2000, **torus),
        # bounded-degree graphs of the precision study: 3-regular in binary32, 4-regular in binary16
        dict(name="trial_reg3_20k_f32", kind="trial", graph="regular", n=20000, d=3, storage="f32",
             replicas=2048, sweeps=500, **graph),
        dict(name="trial_reg4_10k_f16", kind="trial", graph="regular", n=10000, d=4, storage="f16",
             replicas=2048, sweeps=500, **graph),
        # a weighted sparse graph of odd size, coloured greedily by the library
        dict(name="trial_gnm10k_f32", kind="trial", graph="gnm", n=9973, m=24931, wmax=3, storage="f32",
             replicas=256, sweeps=1000, **graph),
        # local fields with tracking and drawn twist directions on a weighted lattice (QUBO-like input)
        dict(name="fields_torus10k_f32", kind="fields", graph="torus2d", L1=100, L2=100, wmax=2, storage="f32",
             replicas=1024, sweeps=500, track=125, alpha0=25.0, ratio=1.0, period=3),
        # a ragged batch in one run: tori and weighted sparse graphs, 64-256 trials each
        dict(name="batch_ragged48_f32", kind="batch", count=48, n_lo=800, n_hi=20000, storage="f32",
             sweeps=200, **graph),
        # serving: requests on 2D and 3D lattices through the server, 32 trials each
        dict(name="serve_lattices_f16", kind="serve", count=12, n_lo=1000, n_hi=50000, storage="f16",
             replicas=32, sweeps=500, alpha0=25.0, ratio=1.0, period=3),
        # the optimal-bisector readout of a kept state (trials of any age: spread out to settled phases)
        dict(name="readout_opt_torus20k", kind="readout", graph="torus2d", L1=100, L2=200, storage="f32",
             replicas=512, **torus),
        # a trial checkpointed halfway and resumed: state out, state in, the rest of the anneal
        dict(name="resume_torus20k_f32", kind="resume", graph="torus2d", L1=100, L2=200, storage="f32",
             replicas=256, sweeps=400, **torus),
    ]


# ---------------------------------------------------------------- graphs
class Graph:
    """What the binding takes as an instance: n, src, dst, w, dims."""

    def __init__(self, n, a, b, w, dims=()):
        self.n = int(n)
        self.src = np.minimum(a, b).astype(np.int32)
        self.dst = np.maximum(a, b).astype(np.int32)
        self.w = np.asarray(w, dtype=np.int32)
        self.dims = tuple(int(x) for x in dims)

    @property
    def m(self):
        return int(self.src.shape[0])


def weights(rng, m, wmax):
    w = rng.integers(1, wmax + 1, m)
    return np.where(rng.integers(0, 2, m) == 0, -w, w)


def torus(rng, dims, wmax=1):
    n = int(np.prod(dims))
    ids = np.arange(n).reshape(dims)
    a = np.concatenate([ids.ravel()] * len(dims))
    b = np.concatenate([np.roll(ids, -1, axis=k).ravel() for k in range(len(dims) - 1, -1, -1)])
    return Graph(n, a, b, weights(rng, a.shape[0], wmax), dims)


def regular(rng, n, d):
    """Random simple d-regular graph: a random pairing, loops and repeated pairs switched away."""
    p = rng.permutation(np.repeat(np.arange(n, dtype=np.int64), d))
    a, b = p[0::2].copy(), p[1::2].copy()
    for _ in range(1000):
        key = np.minimum(a, b) * n + np.maximum(a, b)
        _, first = np.unique(key, return_index=True)
        bad = np.ones(a.shape[0], dtype=bool)
        bad[first] = False
        bad |= a == b
        if not bad.any():
            break
        for e in np.flatnonzero(bad):
            f = int(rng.integers(a.shape[0]))
            b[e], b[f] = b[f], b[e]
    order = np.argsort(np.minimum(a, b) * n + np.maximum(a, b))
    return Graph(n, a[order], b[order], weights(rng, a.shape[0], 1))


def gnm(rng, n, m, wmax):
    key = np.empty(0, dtype=np.int64)
    while key.shape[0] < m:
        a, b = rng.integers(0, n, 2 * m), rng.integers(0, n, 2 * m)
        ok = a != b
        key = np.unique(np.concatenate([key, np.minimum(a, b)[ok] * n + np.maximum(a, b)[ok]]))
    key = np.sort(rng.permutation(key)[:m])
    return Graph(n, key // n, key % n, weights(rng, m, wmax))


def graph_of(case, rng):
    if case["graph"] == "torus2d":
        return torus(rng, (case["L1"], case["L2"]), case.get("wmax", 1))
    if case["graph"] == "regular":
        return regular(rng, case["n"], case["d"])
    return gnm(rng, case["n"], case["m"], case["wmax"])


def sizes(case):
    """(n, m) of a single-graph case."""
    if case["graph"] == "torus2d":
        n = case["L1"] * case["L2"]
        return n, 2 * n
    if case["graph"] == "regular":
        return case["n"], case["n"] * case["d"] // 2
    return case["n"], case["m"]


def even_near(x):
    return max(4, 2 * int(round(x / 2)))


def many(case):
    """The instances of a batch or a serving case: kind, sizes and replicas of each, the same for every
    seed (they are part of the case); N evenly spread over the logarithm of its range."""
    out, span = [], math.log(case["n_hi"] / case["n_lo"])
    for k in range(case["count"]):
        n = case["n_lo"] * math.exp(span * (((k * 7) % case["count"]) + 0.5) / case["count"])
        if k % 2 == 0:
            L1 = even_near(math.sqrt(n))
            dims = (L1, even_near(n / L1))
        elif case["kind"] == "serve":
            L1 = even_near(n ** (1 / 3))
            L2 = even_near(math.sqrt(n / L1))
            dims = (L1, L2, even_near(n / L1 / L2))
        else:
            dims = ()
        n = int(np.prod(dims)) if dims else int(n) | 1
        m = len(dims) * n if dims else int(n * (2.0 + ((k * 5) % 11) / 10.0))
        out.append(dict(n=n, m=m, dims=dims, replicas=64 + (k * 37) % 193 if case["kind"] == "batch"
                        else case["replicas"]))
    return out


# ---------------------------------------------------------------- cases of the same ranges
def between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the kinds of listed(), sizes over their whole range, every storage form."""
    kind = rng.choice(["trial_torus", "trial_torus", "trial_regular", "trial_gnm", "solve", "fields", "batch",
                       "serve", "readout", "resume"])
    case = dict(storage=rng.choice(["f32", "f32", "f16", "q16", "bf16"]), period=rng.choice([3, 3, 6]),
                ratio=rng.choice([0.5, 1.0]), alpha0=rng.choice([14.0, 14.0, 25.0]))
    if kind == "batch":
        case.update(kind="batch", count=between(rng, 4, 48), n_lo=800, n_hi=between(rng, 2000, 20000),
                    sweeps=between(rng, 50, 200))
        return case
    if kind == "serve":
        case.update(kind="serve", count=between(rng, 1, 12), n_lo=1000, n_hi=between(rng, 2000, 50000),
                    replicas=rng.choice([16, 32, 32, 50]), sweeps=between(rng, 100, 500))
        return case
    case["replicas"] = between(rng, 64, 2048)
    if kind in ("trial_torus", "solve", "fields", "readout", "resume"):
        case.update(graph="torus2d", L1=even_near(between(rng, 16, 100)), L2=even_near(between(rng, 16, 200)))
    elif kind == "trial_regular":
        case.update(graph="regular", n=2 * between(rng, 250, 10000), d=rng.choice([3, 4, 5]))
    else:
        n = between(rng, 500, 20000)
        case.update(graph="gnm", n=n, m=int(n * rng.uniform(2.0, 3.0)), wmax=rng.choice([1, 3, 3, 7]))
    case["kind"] = "trial" if kind.startswith("trial") else kind
    n, m = sizes(case)
    if kind == "readout":
        case["replicas"] = max(1, min(case["replicas"], 512 * 20000 // n))
        return case
    most = MOST_UPDATES // 4
    if kind == "fields":
        case.update(wmax=rng.choice([1, 2, 3]), alpha0=25.0)
        most = 20000 * 1024 * 500
    if kind == "resume":
        case["replicas"] = max(1, min(case["replicas"], 256 * 20000 // n))
        most = 40000 * 256 * 400
    case["sweeps"] = max(20, min(between(rng, 200, 2000), most // (m * case["replicas"])))
    case["replicas"] = max(1, min(case["replicas"], most // (m * case["sweeps"])))
    if kind == "fields":
        case["track"] = max(5, case["sweeps"] // 4)
    return case


# ---------------------------------------------------------------- what a program holds before the call
def params(case, flags=0):
    return dict(alpha0_deg=case["alpha0"], dwt_ratio=case["ratio"], dwt_period=case["period"],
                storage=STORAGE[case["storage"]], flags=flags)


def phases_in(case, n, rng):
    """Phases of trials of every age: two antipodal groups around a random axis, spread from settled to
    uniform over the replicas, on the 2^-16-turn grid (so every storage but the two 16-bit floats holds
    them exactly)."""
    R = case["replicas"]
    spread = np.exp(np.linspace(math.log(2e-3), math.log(0.5), R))[:, None]
    x = rng.random((R, 1)) + 0.5 * rng.integers(0, 2, (R, n)) + spread * (rng.random((R, n)) - 0.5)
    return np.floor(x * 65536.0) % 65536.0 / 65536.0


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    st = dict(case=case, seed=int(rng.integers(1, 2 ** 62)))
    if case["kind"] == "batch":
        st["what"] = many(case)
        gs = [torus(rng, i["dims"]) if i["dims"] else gnm(rng, i["n"], i["m"], 3) for i in st["what"]]
        st["batch"] = cosm.Batch(gs, **params(case))
        st["replicas"] = [i["replicas"] for i in st["what"]]
        st["seeds"] = rng.integers(1, 2 ** 62, len(gs)).astype(np.uint64)
        return st
    if case["kind"] == "serve":
        st["graphs"] = [torus(rng, i["dims"]) for i in many(case)]
        st["server"] = cosm.Server(memory_budget=8 << 30, max_active=64, chunk_sweeps=500)
        st["params"] = cosm.default_params(**params(case))
        return st
    g = graph_of(case, rng)
    st["graph"] = g
    if case["kind"] == "solve":
        return st
    if case["kind"] == "fields":
        h = np.where(rng.random(g.n) < 0.1, rng.choice([-1, 1], g.n), 0)
        prm = cosm.default_params(track_period=case["track"], **params(case, cosm.DWT_RANDOM_DIR))
        st["solver"] = cosm.Solver(g.n, g.src, g.dst, g.w, dims=g.dims, params=prm, h=h)
        return st
    if case["graph"] == "regular":
        col, nc = cosm.color_misra_gries(g.n, g.src, g.dst)
        st["solver"] = cosm.Solver.from_instance(g, color=col, n_colors=nc, **params(case))
    else:
        st["solver"] = cosm.Solver.from_instance(
            g, **params(case, cosm.OPT_BISECTOR if case["kind"] == "readout" else 0))
    if case["kind"] == "readout":
        st["solver"].set_state(phases_in(case, g.n, rng), seed=st["seed"])
    return st


# ---------------------------------------------------------------- one pass
def results(s):
    """What a program takes from a solver after a run: the best replica and every replica's cut."""
    cut, energy, replica, spins = s.best()
    cuts, bisectors = s.replica_cuts()
    return dict(cut=cut, energy=energy, replica=replica, spins=spins, cuts=cuts, bisectors=bisectors)


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "trial":
        st["solver"].run(case["sweeps"], case["replicas"], st["seed"])
        return results(st["solver"])
    if kind == "solve":
        g = st["graph"]
        cut, energy, spins, cuts = cosm.solve(g.n, g.src, g.dst, g.w, case["sweeps"], case["replicas"], st["seed"],
                                              dims=g.dims, replica_cuts=True, **params(case))
        return dict(cut=cut, energy=energy, spins=spins, cuts=cuts)
    if kind == "fields":
        s = st["solver"]
        s.run(case["sweeps"], case["replicas"], st["seed"])
        return dict(results(s), energies=s.replica_energies(), trace=s.trace())
    if kind == "batch":
        b = st["batch"]
        b.run(case["sweeps"], st["replicas"], st["seeds"])
        b.sync()
        best = [b.best(i) for i in range(len(st["replicas"]))]
        return dict(cut=np.array([x[0] for x in best]), energy=np.array([x[1] for x in best]),
                    replica=np.array([x[2] for x in best]), spins=np.concatenate([x[3] for x in best]),
                    cuts=np.concatenate([b.replica_cuts(i)[0] for i in range(len(best))]))
    if kind == "serve":
        srv = st["server"]
        # a target no cut reaches: every request takes one whole trial
        ids = [srv.submit(g, case["sweeps"], case["replicas"], st["seed"] + k, 1 << 40, max_trials=1,
                          params=st["params"]) for k, g in enumerate(st["graphs"])]
        done = [srv.wait(i, timeout=60.0) for i in ids]
        return dict({k: np.array([d[k] for d in done]) for k in ("status", "best_cut", "energy", "best_trial",
                                                                 "best_replica")},
                    spins=np.concatenate([srv.spins(i) for i in ids]))
    if kind == "readout":
        s = st["solver"]
        s.readout()
        return dict(results(s), energies=s.replica_energies(), positions=s.replica_bisectors())
    # resume: half the anneal, the state out and in again, the other half
    s, S, R = st["solver"], case["sweeps"], case["replicas"]
    s.run_range(S, 1, S // 2, R, st["seed"])
    phases, at = s.export_state()
    s.import_state(phases, R, st["seed"], at)
    s.run_range(S, at + 1, S, R, st["seed"])
    return dict(results(s), phases=phases, at=at)


# ---------------------------------------------------------------- what a pass cannot do without
def trial_work(n, m, replicas, sweeps, period):
    """Graph in, results out; per edge, replica and sweep the difference, its sign and two phase updates,
    per vertex, replica and twist the window test and the update."""
    flops = replicas * sweeps * (4.0 * m + (2.0 * n / period if period else 0.0))
    return dict(bytes=12.0 * m + n + 12.0 * replicas, flops=flops)


def work(case):
    if case["kind"] in ("batch", "serve"):
        ws = [trial_work(i["n"], i["m"], i["replicas"], case["sweeps"], case["period"]) for i in many(case)]
        return dict(bytes=sum(w["bytes"] for w in ws), flops=sum(w["flops"] for w in ws))
    n, m = sizes(case)
    R = case["replicas"]
    width = 4.0 if case["storage"] == "f32" else 2.0
    if case["kind"] == "readout":
        # the state in, one position per replica out; a comparison per vertex and level of a sort
        return dict(bytes=R * n * width + 12.0 * m + n + 28.0 * R, flops=R * (3.0 * m + n * math.log2(n)))
    w = trial_work(n, m, R, case["sweeps"], case["period"])
    if case["kind"] == "resume":
        w["bytes"] += 2.0 * R * n * width
    if case["kind"] == "fields":
        w["bytes"] += 4.0 * n + 8.0 * R * (2 + -(-case["sweeps"] // case["track"]))
        w["flops"] += 3.0 * n * R * case["sweeps"]
    return w


# ---------------------------------------------------------------- 64-bit values
def exact(case, seed):
    """The outputs of a readout from whole-number arithmetic on the given phases: the best cut over every
    bisector of the 2^32-point circle (the smallest position on ties). Trials have no such value."""
    if case["kind"] != "readout" or case["storage"] in ("f16", "bf16"):
        return None
    rng = np.random.default_rng(seed)
    rng.integers(1, 2 ** 62)
    g = graph_of(case, rng)
    x = torch.from_numpy(phases_in(case, g.n, rng))
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    src, dst = torch.from_numpy(g.src).long().to(dev), torch.from_numpy(g.dst).long().to(dev)
    w = torch.from_numpy(g.w).long().to(dev)
    W = int(g.w.astype(np.int64).sum())
    cuts, where, all_q = [], [], []
    for r in range(case["replicas"]):
        q = (x[r].to(dev) * 4294967296.0).floor().long()
        pos, side = q & 0x7FFFFFFF, q >> 31
        crossed = side[src] != side[dst]
        c0 = int(w[crossed].sum())
        d = torch.where(crossed, -w, w)
        lo, hi = torch.minimum(pos[src], pos[dst]), torch.maximum(pos[src], pos[dst])
        # the cut changes by d just after lo and back just after hi
        at = torch.cat([lo, hi])
        by = torch.cat([d, -d])
        places, inverse = torch.unique(at, return_inverse=True)
        change = torch.zeros(places.shape[0], dtype=torch.int64, device=dev).index_add_(0, inverse, by)
        level = c0 + torch.cumsum(change, 0)
        level = torch.where(places + 1 < 0x80000000, level, torch.full_like(level, -(1 << 62)))
        top = int(level.max())
        if top > c0:
            cuts.append(top)
            where.append(int(places[level == top].min()) + 1)
        else:
            cuts.append(c0)
            where.append(0)
        all_q.append(q.cpu())
    cuts, where = np.array(cuts, dtype=np.int64), np.array(where, dtype=np.int64)
    best = int(np.argmax(cuts))
    spins = np.where(((all_q[best].numpy() - where[best]) & 0xFFFFFFFF) < 0x80000000, 1, -1).astype(np.int8)
    return dict(cut=int(cuts[best]), energy=W - 2 * int(cuts[best]), replica=best, spins=spins, cuts=cuts,
                bisectors=np.full(cuts.shape[0], -1, dtype=np.int32), energies=W - 2 * cuts,
                positions=where.astype(np.uint32))
