"""Edge lists on record tables: whole trials equal the plain records bit for bit,
for every record format, tile width and rows per warp -- colours of every size
(empty places in a last row, warps without rows), one warp to 32."""
import os

import numpy as np
import pytest

import instances

pytestmark = pytest.mark.gpu

GRAPHS = {
    "tiny": lambda: instances.sparse_gnm(5, 4, 1),
    "signs": lambda: instances.sparse_gnm(701, 2100, 5, wmax=1),
    "packed": lambda: instances.sparse_gnm(1000, 2600, 5),         # |w| <= 3
    "offsets": lambda: instances.sparse_gnm(333, 900, 5, wmax=63),  # two words
    "plain": lambda: instances.sparse_gnm(333, 900, 5, wmax=100),   # float forms keep the plain records
}


def trial(cosm, inst, env, replicas, **kw):
    os.environ.update(env)
    try:
        s = cosm.Solver(inst.n, inst.src, inst.dst, inst.w, **kw)
        s.run(41, replicas, seed=5)
        out = [s.export_state()[0], *s.replica_cuts(), s.best()[3], s.replica_energies()]
        return out + ([s.trace()] if kw.get("track_period") else [])
    finally:
        for k in env:
            os.environ.pop(k, None)


@pytest.mark.parametrize("storage,K", [(0, 1), (0, 2), (0, 4), (1, 2), (1, 4), (1, 8), (2, 2), (2, 4), (2, 8),
                                       (3, 2), (3, 8)])
@pytest.mark.parametrize("graph", GRAPHS)
def test_tables_equal_plain_records(storage, K, graph):
    import paper_2605_30355_gb300 as cosm
    inst = GRAPHS[graph]()
    h = instances.Stream(3).below(5, inst.n) - 2
    variants = [dict(dwt_ratio=1.0),
                dict(dwt_ratio=1.0, flags=cosm.DWT_RANDOM_DIR, track_period=7, n_bisectors=5),
                dict(alpha0_deg=100.0, dwt_period=1),  # every binary32 update wrapped
                dict(dwt_period=0), dict(dwt_ratio=1.0, h=h)]
    for kw in variants:
        base = trial(cosm, inst, {"COSM_K": str(K), "COSM_SPLIT_W": "1"}, 2 * K + 1, storage=storage, **kw)
        for threads in ("32", "96", "512"):
            got = trial(cosm, inst, {"COSM_K": str(K), "COSM_THREADS": threads}, 2 * K + 1, storage=storage, **kw)
            for a, b in zip(base, got):
                assert np.array_equal(a, b), (kw, threads)
