"""2D lattices with their phases in registers: whole trials equal the passes on
shared memory bit for bit, for every patch shape and tile width, at sides that
the shapes divide and sides that leave short patches at the ends."""
import os

import numpy as np
import pytest

import instances

pytestmark = pytest.mark.gpu

SHAPES = [(2, 5), (2, 4), (2, 3), (2, 2), (1, 2), (1, 1)]


def fits(blocks, most):
    grid = -(-blocks // most)
    missing = grid * most - blocks
    return missing <= grid and not (most == 1 and missing)


def trial(cosm, inst, env, replicas, sweeps, **kw):
    os.environ.update(env)
    try:
        s = cosm.Solver.from_instance(inst, **kw)
        s.run(sweeps, replicas, seed=5)
        out = [s.export_state()[0], *s.replica_cuts(), s.best()[3], s.replica_energies()]
        if kw.get("track_period"):
            out.append(s.trace())
        return out, s.layout()
    finally:
        for k in env:
            os.environ.pop(k, None)


@pytest.mark.parametrize("storage,K", [(0, 2), (1, 2), (1, 4), (2, 2), (2, 4), (3, 2), (3, 4)])
@pytest.mark.parametrize("dims", [(4, 4), (4, 6), (10, 14), (16, 16), (20, 22), (30, 34), (46, 58)])
def test_registers_equal_shared_memory(storage, K, dims):
    import paper_2605_30355_gb300 as cosm
    inst = instances.torus2d(*dims, 1)
    variants = [dict(dwt_ratio=0.5), dict(dwt_ratio=1.0, flags=cosm.DWT_RANDOM_DIR, track_period=7),
                dict(alpha0_deg=40.0, dwt_period=1, flags=cosm.DWT_RANDOM_DIR, n_bisectors=3)]
    for kw in variants:
        base, _ = trial(cosm, inst, {"COSM_PATCH": "-1", "COSM_K": str(K)}, 2 * K + 1, 61, storage=storage, **kw)
        for i, (r, c) in enumerate(SHAPES):
            if not fits(dims[0] // 2, r) or not fits(dims[1] // 2, c):
                continue
            env = {"COSM_PATCH": str(i), "COSM_K": str(K)}
            got, lay = trial(cosm, inst, env, 2 * K + 1, 61, storage=storage, **kw)
            assert lay["lattice"] == 2 and lay["K"] == K
            for a, b in zip(base, got):
                assert np.array_equal(a, b), (kw, (r, c))


@pytest.mark.parametrize("storage", [0, 2])
def test_registers_in_the_wraparound_schedule_and_ranges(storage):
    # split tiles hand their state over through global memory; ranges store
    # and load it between launches
    import paper_2605_30355_gb300 as cosm
    inst = instances.torus2d(22, 26, 3)
    whole, _ = trial(cosm, inst, {"COSM_PATCH": "-1"}, 37, 90, storage=storage)
    split, lay = trial(cosm, inst, {"COSM_GRID_CAP": "5"}, 37, 90, storage=storage)
    assert lay["grid"] == 5
    s = cosm.Solver.from_instance(inst, storage=storage)
    s.run_range(90, 1, 31, 37, 5)
    s.run_range(90, 32, 90, 37, 5)
    ranges = [s.export_state()[0], *s.replica_cuts(), s.best()[3], s.replica_energies()]
    for got in (split, ranges):
        for a, b in zip(whole, got):
            assert np.array_equal(a, b)
