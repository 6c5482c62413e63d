"""Building an instance: edges may come in any order (the device tables and so
whole trials are the same), a duplicate is refused wherever it stands, and
requests that a server admits together get the results they get alone."""
import numpy as np
import pytest

import instances

pytestmark = pytest.mark.gpu


def graph(kind):
    return {"torus2d": lambda: instances.torus2d(10, 14, 3), "torus3d": lambda: instances.torus3d(4, 6, 8, 3),
            "gnm": lambda: instances.sparse_gnm(301, 700, 3)}[kind]()


@pytest.mark.parametrize("kind", ["torus2d", "torus3d", "gnm"])
def test_edge_order_changes_nothing(kind):
    import paper_2605_30355_gb300 as cosm
    g = graph(kind)
    color, C = cosm.color_greedy(g.n, g.src, g.dst) if kind == "gnm" else (None, 0)
    out = []
    for order in (np.arange(g.m), np.random.default_rng(1).permutation(g.m), np.arange(g.m)[::-1]):
        s = cosm.Solver(g.n, g.src[order], g.dst[order], g.w[order], dims=g.dims,
                        color=None if color is None else color[order], n_colors=C)
        s.run(60, 6, seed=5)
        out.append([s.export_state()[0], *s.replica_cuts(), s.best()[3]])
    for other in out[1:]:
        for a, b in zip(out[0], other):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("at", [0, 1, 350, 699, 700])
def test_duplicate_refused_anywhere(at):
    import paper_2605_30355_gb300 as cosm
    g = graph("gnm")
    for of in (0, g.m - 1):
        src, dst, w = (np.insert(x, at, x[of]) for x in (g.src, g.dst, g.w))
        with pytest.raises(Exception, match="duplicate"):
            cosm.Solver(g.n, src, dst, w)


@pytest.mark.parametrize("count", [2, 20])
def test_requests_admitted_together(count):
    import paper_2605_30355_gb300 as cosm
    reqs = [(instances.torus2d(40, 60, 1), 4000)]  # keeps the server busy while the others queue
    reqs += [(graph(("torus2d", "torus3d", "gnm")[k % 3]), 50 + k) for k in range(count)]
    keys = ("status", "trials", "best_cut", "energy", "best_trial", "best_replica")

    def submit(srv, k):
        return srv.submit(reqs[k][0], reqs[k][1], 8, 7 + k, 1 << 40, storage=k % 2)

    srv = cosm.Server(chunk_sweeps=1000)
    ids = [submit(srv, k) for k in range(len(reqs))]
    mixed = [(srv.wait(i), srv.spins(i)) for i in ids]
    srv.close()
    for k, (res, spins) in enumerate(mixed):
        srv = cosm.Server(chunk_sweeps=1000)
        i = submit(srv, k)
        alone = srv.wait(i)
        np.testing.assert_array_equal(spins, srv.spins(i))
        srv.close()
        assert [res[x] for x in keys] == [alone[x] for x in keys]
