"""The optimal-bisector readout's sort at the sizes where it can go wrong: fewer
vertices than threads or warps, chunks with remainders, the shared-memory and
the global-memory form, every digit of the positions in use or none."""
import numpy as np
import pytest

import instances

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(2, 1), (31, 60), (33, 64), (1023, 2500), (1025, 2500), (8193, 20000),
                                 (24000, 60000), (30011, 70000)])
@pytest.mark.parametrize("storage", [0, 2])
def test_positions_of_every_kind(n, m, storage):
    import oracle as orc
    import paper_2605_30355_gb300 as cosm
    inst = instances.sparse_gnm(n, m, 3)
    s = cosm.Solver(inst.n, inst.src, inst.dst, inst.w, storage=storage, flags=cosm.OPT_BISECTOR)
    g = orc.coloured(inst)
    rng = np.random.default_rng(n)
    u = rng.random((6, n))
    x = np.stack([u[0], np.floor(u[1] * 16) / 16,            # all digits; the top one only
                  0.3 + u[2] * 2.0 ** -20 + 0.5 * (u[3] < 0.5),  # two tight groups: the low digits
                  np.full(n, 0.75), np.floor(u[4] * 2 ** 16) / 2 ** 16, np.where(u[5] < 0.5, 0.0, 0.5)])
    s.set_state(x)
    s.readout()
    y = s.get_state()
    cuts, _ = s.replica_cuts()
    B = s.replica_bisectors()
    for r in range(x.shape[0]):
        c, b, _ = orc.binarize_opt(g, y[r])
        assert (cuts[r], B[r]) == (c, b), r
