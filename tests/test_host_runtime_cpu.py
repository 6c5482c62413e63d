"""The host runtime without a GPU: its own sources linked with a stand-in for
the CUDA runtime and the kernels (fake_device.cpp), which checks every launch
for copies still on their way, for tables of another layout and for states
read in another layout than they were written in."""
import ctypes as C
import importlib.util
import os
import subprocess
import sys
import time

import numpy as np
import pytest

import instances

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2605_30355_gb300")
STREAM = 0x50  # a caller's stream


def build_fake(out):
    sys.path.insert(0, ROOT)
    from paper_2605_30355_gb300 import build
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    src = [os.path.join(ROOT, "tests", "fake_device.cpp")] + \
        [os.path.join(PKG, "csrc", f) for f in ("cosm_runtime.cu", "cosm_server.cu", "cosm_graph.cpp")]
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-w", "-I", os.path.join(PKG, "csrc"), "-I",
                           os.path.join(ROOT, "include"), "-I", cuda, "-x", "c++"] + src +
                          ["-o", out, "-static-libstdc++", "-static-libgcc", "-Wl,-Bsymbolic", "-ldl", "-lpthread"])
    return out


def load_fake(path):
    """A second copy of the package, bound to the library at `path`."""
    spec = importlib.util.spec_from_file_location("cosm_on_fake", os.path.join(PKG, "__init__.py"),
                                                  submodule_search_locations=[PKG])
    cosm = importlib.util.module_from_spec(spec)
    sys.modules["cosm_on_fake"] = cosm
    spec.loader.exec_module(cosm)
    cosm.LIB_PATH = path
    lib = cosm.lib()
    lib.fake_message.restype = C.c_char_p
    lib.fake_peak_bytes.restype = C.c_int64
    lib.fake_fail_malloc.argtypes = [C.c_int64]
    return cosm


@pytest.fixture(scope="session")
def fake_path(tmp_path_factory):
    return build_fake(str(tmp_path_factory.mktemp("fake") / "libcosm_host.so"))


@pytest.fixture
def cosm(fake_path):
    cosm = load_fake(fake_path)
    report(cosm)
    return cosm


def report(cosm):
    """What the launches since the last report were, and what was wrong with them."""
    out = (C.c_int64 * 8)()
    msg = cosm.lib().fake_message().decode()
    cosm.lib().fake_report(out)
    return dict(zip(("unordered", "bad", "launches", "threads", "K", "shape", "ragged", "format"), out), message=msg)


def sound(cosm):
    r = report(cosm)
    assert r["bad"] == 0 and r["unordered"] == 0, r
    return r


GRAPHS = {"edges": lambda: instances.sparse_gnm(900, 2400, 1), "lattice": lambda: instances.torus2d(40, 60, 1)}


@pytest.mark.parametrize("graph", GRAPHS)
def test_uploads_arrive_before_launches_on_other_streams(cosm, graph):
    # a copy from pageable memory may still be queued on the legacy stream when
    # cudaMemcpy returns; streams created non-blocking do not wait for it
    inst = GRAPHS[graph]()
    s = cosm.Solver.from_instance(inst)
    for replicas in (4, 4096, 4):  # a new layout each time
        s.run(20, replicas, 1, stream=STREAM)
        sound(cosm)
    s.set_state(np.zeros((4, inst.n)))
    s.step(1, 0.01, stream=STREAM)
    s.import_state(s.export_state()[0], 4, 1, 5)
    s.run_range(20, 6, 20, 4, 1, stream=STREAM)
    s.readout(stream=STREAM)
    sound(cosm)


def test_batch_and_server_uploads_arrive_before_their_launches(cosm):
    insts = [g() for g in GRAPHS.values()] * 3
    b = cosm.Batch(insts)
    b.run(20, 4, 1)
    sound(cosm)
    b.run(20, 4096, 1)  # other layouts
    sound(cosm)
    srv = cosm.Server(chunk_sweeps=7)
    for rid in [srv.submit(inst, 20, 4, 1, 10 ** 9) for inst in insts]:
        assert srv.wait(rid, 60)["status"] == cosm.EXHAUSTED
    srv.close()
    sound(cosm)


@pytest.mark.parametrize("entry", ["run", "set_state", "import_state"])
@pytest.mark.parametrize("graph", GRAPHS)
def test_failed_tables_leave_the_layout_of_the_state(cosm, graph, entry):
    # a run whose tables do not fit in device memory changes nothing: the
    # earlier run's state and results stay readable, and its replica count runs
    # again on its own kernel and table
    inst = GRAPHS[graph]()
    s = cosm.Solver.from_instance(inst)
    s.run(20, 4, 1)
    first = sound(cosm)
    lay = s.layout()
    cosm.lib().fake_fail_malloc(1)
    many = 4096
    with pytest.raises(cosm.CosmError) as err:
        if entry == "run":
            s.run(20, many, 1)
        elif entry == "set_state":
            s.set_state(np.zeros((many, inst.n)))
        else:
            s.import_state(np.zeros((many, inst.n), np.float32), many, 1, 0)
    assert err.value.code == cosm.ERR_NOMEM
    s.replicas = 4
    assert s.layout() == lay
    s.export_state()
    s.replica_cuts()
    s.readout()
    s.run(20, 4, 1)
    again = sound(cosm)
    assert [again[k] for k in ("K", "threads", "shape", "format")] == \
        [first[k] for k in ("K", "threads", "shape", "format")]
    # with memory there, the larger run takes another layout, which is what
    # the failure must not leave behind
    s.run(20, many, 1)
    other = sound(cosm)
    assert [other[k] for k in ("K", "threads", "shape")] != [first[k] for k in ("K", "threads", "shape")]
    s.run(20, 4, 1)
    sound(cosm)


@pytest.mark.parametrize("nth", range(2, 8))
def test_failed_buffers_end_the_state(cosm, nth):
    # the state's buffer may be gone or of another layout: no call reads it
    s = cosm.Solver.from_instance(GRAPHS["edges"]())
    s.run(20, 4, 1)
    sound(cosm)
    cosm.lib().fake_fail_malloc(nth + 2)  # the table's three buffers, then those of the run
    with pytest.raises(cosm.CosmError) as err:
        s.run(20, 4096, 1)
    assert err.value.code == cosm.ERR_NOMEM
    for call in (s.export_state, s.replica_cuts, s.readout, lambda: s.step(1, 0.01)):
        with pytest.raises(cosm.CosmError) as err:
            call()
        assert err.value.code == cosm.ERR_STATE
    s.run(20, 4, 1)
    s.export_state()
    sound(cosm)


def test_failed_batch_run_ends_the_batch_state(cosm):
    insts = [g() for g in GRAPHS.values()]
    b = cosm.Batch(insts)
    b.run([20, 20], [4, 4], [1, 2])
    for bad in (0, 1 << 24):  # refused arguments change nothing
        with pytest.raises(cosm.CosmError) as err:
            b.run([20, 20], [4096, bad], [1, 2])
        assert err.value.code == cosm.ERR_INVALID_ARG
    b.replicas = [4, 4]
    b.get_state(0)
    sound(cosm)
    cosm.lib().fake_fail_malloc(1)
    with pytest.raises(cosm.CosmError) as err:
        b.run([20, 20], [4096, 4096], [1, 2])
    assert err.value.code == cosm.ERR_NOMEM
    b.replicas = [4, 4]
    for call in (b.get_state, b.best, b.replica_cuts):
        with pytest.raises(cosm.CosmError) as err:
            call(0)
        assert err.value.code == cosm.ERR_STATE
    b.run([20, 20], [4096, 4096], [1, 2])
    b.get_state(1)
    b.close()
    assert report(cosm)["bad"] == 0


def test_failed_batch_launch_ends_the_batch_state(cosm):
    # the layouts are new, the launch is not made: no state is read in them
    b = cosm.Batch([g() for g in GRAPHS.values()])
    b.run([20, 20], [4, 4], [1, 2])
    cosm.lib().fake_fail_graphs(1)
    with pytest.raises(cosm.CosmError) as err:
        b.run([20, 20], [4096, 4096], [1, 2])
    cosm.lib().fake_fail_graphs(0)
    assert err.value.code == cosm.ERR_CUDA
    b.replicas = [4, 4]
    for call in (b.get_state, b.best, b.replica_cuts):
        with pytest.raises(cosm.CosmError) as err:
            call(0)
        assert err.value.code == cosm.ERR_STATE
    b.run([20, 20], [4, 4], [1, 2])
    b.get_state(0)
    b.close()
    sound(cosm)


def test_host_threads_that_cannot_be_created(fake_path):
    # the calling thread does the work; in a process of its own, as an escaping
    # exception would end it
    code = """
import sys; sys.path[:0] = [%r, %r]
import test_host_runtime_cpu as T, instances
cosm = T.load_fake(%r)
insts = [g() for g in T.GRAPHS.values()] * 3
lib = cosm.lib()
lib.fake_fail_threads(1)
b = cosm.Batch(insts)
b.run(20, 4, 1)
b.run(20, 4096, 1)
try:
    cosm.Server()
    raise SystemExit("a server without its thread")
except cosm.CosmError as e:
    assert e.code == cosm.ERR_NOMEM
lib.fake_fail_threads(0)
srv = cosm.Server(max_active=16)
lib.fake_fail_threads(1)
ids = [srv.submit(inst, 20, 4, 1, 10 ** 9) for inst in insts]
assert all(srv.wait(rid, 60)["status"] == cosm.EXHAUSTED for rid in ids)
srv.close()
T.sound(cosm)
""" % (ROOT, os.path.join(ROOT, "tests"), fake_path)
    done = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=120)
    assert done.returncode == 0, done.stderr


def test_forced_thread_counts_are_at_least_a_warp(cosm, monkeypatch, tmp_path):
    # the readout's scan of the bisectors takes all 32 lanes
    lattice, edges = GRAPHS["lattice"](), GRAPHS["edges"]()
    srv = cosm.Server(threads=8)
    for kw in (dict(flags=cosm.NO_SCS), dict()):
        for inst in (lattice, edges):
            rid = srv.submit(inst, 20, 4, 1, 10 ** 9, **kw)
            assert srv.wait(rid, 60)["status"] == cosm.EXHAUSTED
            assert sound(cosm)["threads"] >= 32
    srv.close()
    monkeypatch.setenv("COSM_THREADS", "8")
    for inst in (lattice, edges):
        s = cosm.Solver.from_instance(inst)
        s.run(20, 4, 1)
        assert s.layout()["threads"] == 32
        sound(cosm)
    monkeypatch.delenv("COSM_THREADS")
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("COSM_TUNE_CACHE", str(cache))
    for kw in (dict(flags=cosm.NO_SCS), dict()):
        cache.write_text("")
        b = cosm.Batch([lattice, edges], **kw)
        b.tune(4)
        key = cache.read_text().split()[0]
        for threads in (8, 40):
            cache.write_text("%s 0 %d\n" % (key, threads))
            b.tune(4)
            b.run(20, 4, 1)
            assert sound(cosm)["threads"] >= 32 and b.info()["threads"] == threads
        b.close()


def _heavier(inst, wmax):
    w = 1 + instances.Stream(9).below(wmax, inst.m)
    return instances.Instance(inst.n, inst.src, inst.dst, np.asarray(w, np.int32), inst.dims)


REQUESTS = {
    "signs": lambda: instances.random_regular(6000, 3, 1),
    "weights": lambda: _heavier(instances.sparse_gnm(5000, 60000, 2), 60),
    "small": lambda: instances.sparse_gnm(60, 100, 3),
    "torus": lambda: instances.torus2d(100, 100, 1),
    "heavy torus": lambda: _heavier(instances.torus2d(60, 60, 1), 50),
    "3D": lambda: instances.torus3d(12, 12, 14, 1),
}


@pytest.mark.parametrize("threads", [0, 96])
@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("graph", REQUESTS)
def test_a_request_holds_no_more_than_its_footprint(cosm, graph, storage, threads):
    inst = REQUESTS[graph]()
    lib = cosm.lib()
    for kw in (dict(), dict(alpha0_deg=100.0), dict(flags=cosm.NO_SCS)):
        lib.fake_peak_bytes()
        srv = cosm.Server(threads=threads)
        before = lib.fake_peak_bytes()
        srv.wait(srv.submit(inst, 50, 3, 1, 10 ** 9, storage=storage, **kw), 60)
        held, fp = lib.fake_peak_bytes() - before, srv.stats()["peak_footprint"]
        srv.close()
        sound(cosm)
        assert held <= fp + 1024, kw  # the server's own work lists of a few units
        # what was accepted without counting the tables is accepted, alone
        esz = 4 if storage == 0 else 2
        base = 5 * inst.m + 4 * inst.n + 260 + 3 * (inst.n * esz + 64) + 72 + 400 + inst.n + inst.n // 2 + 4096
        srv = cosm.Server(memory_budget=base, threads=threads)
        ids = [srv.submit(inst, 50, 3, k, 10 ** 9, storage=storage, **kw) for k in range(2)]
        assert all(srv.wait(rid, 60)["status"] == cosm.EXHAUSTED for rid in ids)
        assert srv.stats()["max_concurrent"] == 1 and srv.stats()["peak_footprint"] <= base
        srv.close()
        srv = cosm.Server(memory_budget=base - 1)
        with pytest.raises(cosm.CosmError) as err:
            srv.submit(inst, 50, 3, 1, 10 ** 9, storage=storage, **kw)
        assert err.value.code == cosm.ERR_TOO_LARGE
        srv.close()


def test_tile_policies_differ_and_tuning_keys_name_what_decides_them(cosm, monkeypatch, tmp_path):
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("COSM_TUNE_CACHE", str(cache))

    def key(insts, **kw):
        cache.write_text("")
        b = cosm.Batch(insts, **kw)
        b.tune(64)
        return cache.read_text().split()[0], b

    edges = [instances.sparse_gnm(n, 5 * n // 2, n) for n in (300, 1000, 2500, 5000, 9000)]
    for insts, kw, least in ((edges, dict(), 1), (edges, dict(storage=1), 2), (edges, dict(storage=2), 2),
                             ([instances.torus2d(40, 40, 1)], dict(), 2),
                             ([instances.torus2d(40, 40, 1)], dict(storage=2), 2)):
        k, b = key(insts, **kw)
        widths = {}
        for policy in range(4):
            cache.write_text("%s %d 0\n" % (k, policy))
            b.tune(64)
            b.run(50, 64, 1)
            sound(cosm)
            widths[policy] = [b.layout(i)["K"] for i in range(len(insts))]
        b.close()
        assert widths[1] == [least] * len(insts)
        assert all(x <= y for x, y in zip(widths[3], widths[0]))
        assert insts is not edges or widths[3] != widths[0], widths
    base, _ = key(edges)
    heavier, _ = key(edges[:-1] + [_heavier(edges[-1], 40)])
    others = [key(edges, **kw)[0] for kw in (dict(n_bisectors=7), dict(alpha0_deg=120.0))]
    assert len({base, heavier, *others}) == 4


def test_an_admitted_request_counts_what_it_holds(cosm):
    # two requests whose bounds exceed the budget, not what they hold: the
    # second joins the first once that is admitted
    inst, sweeps = REQUESTS["torus"](), 30000
    lib = cosm.lib()

    def running(srv, count):
        end = time.monotonic() + 30
        while srv.stats()["active"] < count:
            assert time.monotonic() < end

    srv = cosm.Server(chunk_sweeps=1)
    rid = srv.submit(inst, sweeps, 4, 1, 10 ** 9, storage=1)
    running(srv, 1)
    st = srv.stats()
    held, bound = st["footprint"], st["peak_footprint"]
    assert 0 < held < bound
    srv.close()
    srv = cosm.Server(chunk_sweeps=1, memory_budget=held + bound)
    for k in range(2):
        srv.submit(inst, sweeps, 4, k, 10 ** 9, storage=1)
    running(srv, 2)
    assert srv.stats()["peak_footprint"] <= held + bound
    srv.close()
    sound(cosm)


def _weighted(n, m, wmax, seed):
    inst = instances.sparse_gnm(n, m, seed, wmax=wmax)
    w = np.array(inst.w, np.int32)
    w[:2] = wmax, -wmax  # the extremes are there
    return instances.Instance(inst.n, inst.src, inst.dst, w)


# (vertices, largest weight, storage, tile width) -> format: both sides of every
# limit (2^14 and 2^15 slots, the weights a code or two words hold, every
# update wrapped)
FORMATS = [
    ((5, 1, 0, 1), 0), ((700, 1, 0, 4), 0), ((700, 1, 1, 8), 0), ((700, 1, 2, 8), 0),
    ((1 << 15, 1, 0, 1), 0), ((1 << 15, 1, 1, 2), 0), ((1 << 15, 1, 2, 2), 0),
    (((1 << 15) + 1, 1, 0, 1), 2), (((1 << 15) + 1, 1, 1, 2), 2), (((1 << 15) + 1, 1, 2, 2), 2),
    ((700, 2, 0, 1), 2), ((700, 2, 1, 2), 2), ((700, 3, 0, 2), 1), ((700, 3, 1, 4), 1), ((700, 3, 2, 4), 1),
    ((700, 4, 0, 2), 2), ((700, 4, 1, 4), 2), ((700, 4, 2, 4), 2),
    ((700, 7, 0, 4), 1), ((700, 7, 1, 8), 1), ((700, 7, 2, 8), 1), ((700, 8, 0, 4), 2), ((700, 8, 2, 8), 2),
    ((1 << 14, 3, 0, 2), 1), ((1 << 14, 3, 1, 4), 1), (((1 << 14) + 1, 3, 0, 2), 2), (((1 << 14) + 1, 3, 2, 4), 2),
    ((14000, 7, 0, 4), 1), ((14000, 7, 1, 8), 1),  # byte offsets close to 2^18
    ((56000, 63, 0, 1), 2), ((56000, 63, 1, 2), 2), ((56000, 127, 2, 2), 2),
    ((700, 63, 0, 2), 2), ((700, 64, 0, 2), -1), ((700, 64, 3, 2), -1), ((700, 127, 2, 4), 2),
]


@pytest.mark.parametrize("case,fmt", FORMATS)
def test_record_tables_hold_every_edge(cosm, monkeypatch, case, fmt):
    n, wmax, storage, K = case
    inst = _weighted(n, min(n + n // 4, n * (n - 1) // 2), wmax, n)
    monkeypatch.setenv("COSM_K", str(K))
    for kw, each in ((dict(alpha0_deg=0.1), 0), (dict(alpha0_deg=170.0, dwt_period=1), 4 if storage == 0 else 0)):
        want = fmt + each if fmt >= 0 else -1
        if fmt == 0 and each:
            want = 4 + (1 if K > 1 and n <= 1 << 14 else 2)
        for threads in ("32", "96", "1024"):
            monkeypatch.setenv("COSM_THREADS", threads)
            s = cosm.Solver(inst.n, inst.src, inst.dst, inst.w, storage=storage, **kw)
            s.run(3, 2 * K + 1, 1)
            r = sound(cosm)
            assert r["format"] == want and r["K"] == K and r["threads"] == int(threads)
            assert s.layout_form()["format"] == want
            s.close()


def test_a_repeated_batch_run_keeps_its_layouts(cosm):
    lib = cosm.lib()
    lib.fake_queries.restype = C.c_int64
    insts = [g() for g in GRAPHS.values()] * 4
    b = cosm.Batch(insts)
    b.run(20, 4, 1)
    first, info = lib.fake_queries(), b.info()
    b.run(20, 4, 2)
    assert lib.fake_queries() == info["classes"] < first and b.info()["graphs_built"] == 1
    sound(cosm)
    b.run(20, 700, 2)  # other replicas: chosen again
    assert lib.fake_queries() > info["classes"]
    other = [b.layout(i) for i in range(8)]
    c = cosm.Batch(insts)
    c.run(20, 700, 2)
    assert other == [c.layout(i) for i in range(8)]
    sound(cosm)
    lib.fake_fail_malloc(1)
    with pytest.raises(cosm.CosmError):
        b.run(20, 40000, 2)
    b.run(20, 700, 2)
    assert other == [b.layout(i) for i in range(8)]
    b.close()
    c.close()
    sound(cosm)
