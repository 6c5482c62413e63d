"""The kernel that a layout names is the one compared: every patch shape and
record format is pinned by the layout query on both sides of the comparison,
on both sides of the limits where the format changes; a handle that goes from
one replica count to another and back, on a stream of its own, gives what
fresh handles give."""
import os

import numpy as np
import pytest

import instances

pytestmark = pytest.mark.gpu

SHAPES = [(2, 5), (2, 4), (2, 3), (2, 2), (1, 2), (1, 1)]


def trial(cosm, inst, env, replicas, sweeps, **kw):
    os.environ.update(env)
    try:
        s = cosm.Solver(inst.n, inst.src, inst.dst, inst.w, dims=inst.dims, **kw)
        s.run(sweeps, replicas, seed=5)
        return [s.export_state()[0], *s.replica_cuts(), s.best()[3], s.replica_energies()], s.layout_form()
    finally:
        for k in env:
            os.environ.pop(k, None)


def same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


def taken(dims, shape, storage, K):
    """Whether a forced shape has a kernel and fits the lattice."""
    R, C = shape
    grid, ragged = [], False
    for blocks, most in zip((dims[0] // 2, dims[1] // 2), shape):
        g = -(-blocks // most)
        if g * most - blocks > g or (most == 1 and g != blocks):
            return False, False
        ragged |= g * most != blocks
        grid.append(g)
    patches = grid[0] * grid[1]
    site = K * (4 if storage == 0 else 2)
    regs = R * C * site + 45
    most = 512 if regs > 96 else 640 if regs > 80 else 768 if regs > 64 else 1024
    spills = storage in (1, 3) and K == 4 and R * C > 4
    fits = patches * (2 * R + 2 * C - 1) <= dims[0] * dims[1] and (patches + 31) // 32 * 32 <= most
    return fits and not spills, ragged


@pytest.mark.parametrize("storage,K", [(0, 2), (1, 2), (1, 4), (2, 2), (2, 4), (3, 4)])
@pytest.mark.parametrize("dims", [(4, 6), (10, 14), (16, 16), (30, 34), (46, 58), (100, 100)])
def test_forced_patch_shapes_are_the_ones_that_run(storage, K, dims):
    import paper_2605_30355_gb300 as cosm
    inst = instances.torus2d(*dims, 1)
    base, form = trial(cosm, inst, {"COSM_PATCH": "-1", "COSM_K": str(K)}, 2 * K + 1, 13, storage=storage)
    assert form["shape"] == -1
    for i, shape in enumerate(SHAPES):
        got, form = trial(cosm, inst, {"COSM_PATCH": str(i), "COSM_K": str(K)}, 2 * K + 1, 13, storage=storage)
        fits, ragged = taken(dims, shape, storage, K)
        assert (form["shape"], form["ragged"]) == ((i, int(ragged)) if fits else (-1, 0)), shape
        assert same(base, got), shape


# (vertices, largest weight, storage, tile width) -> format
FORMATS = [((1 << 15, 1, 0, 1), 0), (((1 << 15) + 1, 1, 0, 1), 2), ((1 << 15, 1, 1, 2), 0),
           (((1 << 15) + 1, 1, 2, 2), 2), ((1 << 14, 3, 0, 2), 1), (((1 << 14) + 1, 3, 0, 2), 2),
           ((1 << 14, 3, 1, 4), 1), (((1 << 14) + 1, 3, 2, 4), 2), ((14000, 7, 0, 4), 1), ((14000, 7, 2, 8), 1),
           ((56000, 63, 0, 1), 2), ((56000, 63, 1, 2), 2), ((56000, 127, 2, 2), 2)]


@pytest.mark.parametrize("case,fmt", FORMATS)
def test_record_formats_at_their_limits_equal_plain_records(case, fmt):
    import paper_2605_30355_gb300 as cosm
    n, wmax, storage, K = case
    inst = instances.sparse_gnm(n, n + n // 4, n, wmax=wmax)
    w = np.array(inst.w, np.int32)
    w[:2] = wmax, -wmax
    inst = instances.Instance(n, inst.src, inst.dst, w)
    kw = dict(storage=storage, alpha0_deg=0.1, dwt_ratio=1.0)
    base, form = trial(cosm, inst, {"COSM_K": str(K), "COSM_SPLIT_W": "1"}, 2 * K + 1, 7, **kw)
    assert form["format"] == -1
    got, form = trial(cosm, inst, {"COSM_K": str(K)}, 2 * K + 1, 7, **kw)
    assert form["format"] == fmt
    assert same(base, got)


@pytest.mark.parametrize("storage", [0, 2])
@pytest.mark.parametrize("graph", ["edges", "lattice"])
def test_layouts_there_and_back_on_a_stream(graph, storage):
    import torch

    import paper_2605_30355_gb300 as cosm
    inst = instances.sparse_gnm(3000, 8000, 1) if graph == "edges" else instances.torus2d(40, 60, 1)
    st = torch.cuda.Stream()
    s = cosm.Solver.from_instance(inst, storage=storage)
    forms = []
    for replicas in (3, 3000, 3):
        s.run(30, replicas, 7, stream=st)
        forms.append((s.layout(), s.layout_form()))
        got = [s.export_state()[0], *s.replica_cuts(), s.best()[3]]
        fresh = cosm.Solver.from_instance(inst, storage=storage)
        fresh.run(30, replicas, 7)
        assert same(got, [fresh.export_state()[0], *fresh.replica_cuts(), fresh.best()[3]]), replicas
    key = [(f[0]["K"], f[0]["threads"], f[1]["shape"], f[1]["format"]) for f in forms]
    assert key[0] == key[2] and key[0] != key[1]


def test_server_with_few_threads_gives_the_same_results():
    import paper_2605_30355_gb300 as cosm
    insts = [instances.torus2d(20, 24, 1), instances.sparse_gnm(400, 1100, 2)]
    want = None
    for threads in (0, 8, 40):
        srv = cosm.Server(threads=threads)
        ids = [srv.submit(inst, 60, 6, 3, 10 ** 9, flags=f) for inst in insts for f in (0, cosm.NO_SCS)]
        got = [(r["best_cut"], r["best_replica"]) for r in (srv.wait(i, 60) for i in ids)]
        srv.close()
        want = want or got
        assert got == want, threads
