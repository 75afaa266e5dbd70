"""Whole runs in one launch (k_run over the grid, k_tail in one cluster) against the oracle, at the sizes where
they change: a vertex more or less than a thread per vertex, a block, the cluster's capacity; compaction into a
small and into a large graph; reader lists longer than a warp walks alone; limits; a map buffer of odd alignment.
Integer work: everything must be equal."""
import time

import numpy as np
import pytest

import mapgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CAP = 16 * 8704  # vertices the cluster holds


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__

    __graft_entry__.build()
    import paper_0912_2555_gb300 as p

    return p


def compare(pkg, g, flags=0, want=None, runs=2):
    want = want or oracle.run_graph(g)
    h = pkg.map_create(g.n, g.rowptr, g.colidx if g.m else None, pkg.pack_bits(g.acc))
    try:
        for sched in (0, 1) * runs:
            out = torch.full((g.n + 1,), 7, dtype=torch.int32, device="cuda")
            r = pkg.map_run(h, sched=sched, flags=flags, map_out=out[1:])  # 4 bytes off a 16-byte boundary
            assert (r.verdict, r.witness, r.outer) == (want.verdict, want.witness, want.outer), sched
            assert np.array_equal(out[1:].cpu().numpy().view(np.uint32), want.map), sched
            assert int(out[0]) == 7
            if sched == 0:
                assert (r.rounds, r.relaxations, r.inner_iters) == (want.rounds, want.relaxations, want.inner_total)
            else:
                assert all(a <= b for a, b in zip(r.rounds, want.rounds))
    finally:
        pkg.map_destroy(h)


@pytest.mark.parametrize("n", [1, 31, 1023, 1024, 1025, 2049, 8704, 8705, 20000, CAP - 1, CAP, CAP + 1])
def test_sizes_around_the_limits(pkg, n):
    compare(pkg, mapgen.random_graph(n, 1, 6, 0.03, seed=n, variant="plain") if n > 31
            else mapgen.tiny_graph(n, n, max_deg=3, acc_p=0.5), pkg.MAP_FLAG_FRONTIER_START)
    if n > 1000:
        compare(pkg, mapgen.layered_graph(n, max(8, n // 3000), seed=n))


@pytest.mark.parametrize("n,layers,plant", [(400_003, 24, False), (400_003, 24, True), (3_000_001, 180, False),
                                            (CAP * 16, 40, False)])
def test_compaction(pkg, n, layers, plant):
    """Later iterations in the compact graph: in the cluster, or over the grid first (16 % accepting)."""
    compare(pkg, mapgen.layered_graph(n, layers, seed=11, plant=plant, acc_p=0.16 if layers == 40 else 0.01),
            pkg.MAP_FLAG_FRONTIER_START)


@pytest.mark.parametrize("n", [5000, 30_000, CAP + 1000, 700_000])
def test_hubs(pkg, n):
    """Vertices read by thousands of rows beside vertices nobody reads, a chain of values through them."""
    rng = np.random.default_rng(n)
    hubs = rng.choice(n, 3, replace=False)
    deg = rng.integers(0, 3, n)
    rowptr = np.zeros(n + 1, np.uint32)
    np.cumsum(deg, out=rowptr[1:])
    col = rng.integers(0, n, int(rowptr[-1])).astype(np.uint32)
    at = rng.random(col.size) < 0.4
    col[at] = rng.choice(hubs, int(at.sum()))
    acc = (rng.random(n) < 0.02).astype(np.uint8)
    acc[hubs[0]] = 1
    compare(pkg, mapgen.Graph(n, rowptr, col, acc, (0,) * 8, f"hubs-{n}", {}), pkg.MAP_FLAG_FRONTIER_START)


@pytest.mark.parametrize("n,layers", [(3000, 8), (60_000, 30), (500_000, 30)])
def test_limits_and_what_follows(pkg, n, layers):
    """A run stopped by a limit reports the limit, and the next run on the handle is the oracle's."""
    g = mapgen.layered_graph(n, layers, seed=5)
    want = oracle.run_graph(g)
    assert want.outer > 3 and want.rounds[0] > 3
    h = pkg.map_create(g.n, g.rowptr, g.colidx, pkg.pack_bits(g.acc))
    try:
        for sched in (0, 1):
            for kw in (dict(max_outer=1), dict(max_outer=3), dict(max_inner=1), dict(max_inner=2)):
                r = pkg.map_run(h, sched=sched, flags=pkg.MAP_FLAG_FRONTIER_START, allow_limit=True, **kw)
                assert r.status == pkg.MAP_ERR_LIMIT
                assert r.outer == kw.get("max_outer", 1)
                if "max_inner" in kw:
                    assert r.rounds[0] == kw["max_inner"]
                out = np.empty(g.n, np.uint32)
                r = pkg.map_run(h, sched=sched, map_out=out)
                assert (r.verdict, r.witness, r.outer) == (want.verdict, want.witness, want.outer)
                assert np.array_equal(out, want.map)
                if sched == 0:
                    assert (r.rounds, r.relaxations) == (want.rounds, want.relaxations)
    finally:
        pkg.map_destroy(h)
    # the map of a limited synchronous run is the oracle's of that iteration
    lim = oracle.run_graph(g, max_outer=2)
    h = pkg.map_create(g.n, g.rowptr, g.colidx, pkg.pack_bits(g.acc))
    try:
        out = np.empty(g.n, np.uint32)
        pkg.map_run(h, max_outer=2, flags=pkg.MAP_FLAG_FRONTIER_START, map_out=out, allow_limit=True)
        assert np.array_equal(out, lim.map)
    finally:
        pkg.map_destroy(h)


def test_batch_with_compaction(pkg):
    """Graphs that end in different iterations: floods (planted cycles) beside long eliminations."""
    gs = [mapgen.layered_graph(n, max(8, n // 5000), seed=n, plant=bool(i % 3 == 0))
          for i, n in enumerate([1500, 40_000, 200_000, 7001, 90_000, 300_001])]
    gs += [mapgen.tiny_graph(9, 60, max_deg=3, acc_p=0.3), mapgen.from_lists([[1], [0], []], [0, 0, 0])]
    h = pkg.map_batch_create([(g.n, g.rowptr, g.colidx, pkg.pack_bits(g.acc)) for g in gs])
    try:
        for sched in (0, 1):
            out = np.empty(sum(g.n for g in gs), np.uint32)
            rs = pkg.map_batch_run(h, len(gs), sched=sched, flags=pkg.MAP_FLAG_FRONTIER_START, map_out=out)
            off = 0
            for g, r in zip(gs, rs):
                want = oracle.run_graph(g)
                assert (r.verdict, r.witness, r.outer, r.accepting_left >= 0) == (want.verdict, want.witness, want.outer, True)
                assert np.array_equal(out[off:off + g.n], want.map)
                if sched == 0:
                    assert (r.rounds, r.relaxations) == (want.rounds, want.relaxations)
                off += g.n
    finally:
        pkg.map_destroy(h)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.uint32).view(np.int32)).cuda()


@pytest.mark.parametrize("n", [1, 33, 1025, 16385, 65536])
@pytest.mark.parametrize("where", ["device", "host", "rows-host", "entries-host"])
def test_static_set_up(pkg, n, where):
    """map_run_static's set-up in one cluster: readers of a graph with one long row, empty rows and a hub, from
    arrays in either memory, against the oracle."""
    rng = np.random.default_rng(n)
    deg = rng.integers(0, 4, n)
    deg[n // 2] = min(20 * n, 200_000)
    rowptr = np.zeros(n + 1, np.uint32)
    np.cumsum(deg, out=rowptr[1:])
    col = rng.integers(0, n, int(rowptr[-1])).astype(np.uint32)
    col[rng.random(col.size) < 0.2] = n - 1
    g = mapgen.Graph(n, rowptr, col, (rng.random(n) < 0.05).astype(np.uint8), (0,) * 8, "static", {})
    want = oracle.run_graph(g)
    rp = rowptr if where in ("host", "rows-host") else _dev(rowptr)
    ci = col if where in ("host", "entries-host") else _dev(col)
    ab = pkg.pack_bits(g.acc) if where == "host" else _dev(pkg.pack_bits(g.acc))
    for sched in (0, 1):
        out = np.empty(n, np.uint32)
        r = pkg.map_run_static(n, rp, ci, ab, sched=sched, map_out=out)
        assert (r.verdict, r.witness, r.outer, r.edges_total) == (want.verdict, want.witness, want.outer, g.m * want.outer)
        assert np.array_equal(out, want.map)
        if sched == 0:
            assert (r.rounds, r.relaxations) == (want.rounds, want.relaxations)


@pytest.mark.parametrize("rowptr,col,code", [([0, 2, 1], [0, 1], "CSR"), ([0, 1, 2], [0, 2], "CSR"), ([1, 1, 2], [0, 1], "CSR"),
                                             ([0, 1, 600_000], [0, 1], "ARG")])
@pytest.mark.parametrize("on_device", [False, True])
def test_static_refuses_what_it_refused(pkg, rowptr, col, code, on_device):
    to = _dev if on_device else (lambda a: np.array(a, np.uint32))
    out = np.full(2, 9, np.uint32)
    with pytest.raises(pkg.MapError) as e:
        pkg.map_run_static(2, to(rowptr), to(col), to([1]), map_out=out)
    assert e.value.code == getattr(pkg, f"MAP_ERR_{code}")
    assert out.tolist() == [9, 9]


@pytest.mark.parametrize("n", [16384, 16385, 152 * 1024 + 1, 152 * 12288, 152 * 12288 + 1])
def test_sizes_around_the_grid_kernel(pkg, n):
    """k_own between the cluster and k_run: a vertex more than the cluster takes, than a thread holds, and at
    its capacity (12,288 per block on 152 SMs); dense accepting sets, a planted cycle."""
    compare(pkg, mapgen.layered_graph(n, max(8, n // 9000), seed=3), runs=1)
    compare(pkg, mapgen.layered_graph(n, max(8, n // 9000), seed=4, plant=True, acc_p=0.2), runs=1)


@pytest.mark.parametrize("acc_p", [0.001, 0.5, 1.0])
def test_interleaved_products_and_dense_accepting_sets(pkg, acc_p):
    g = mapgen.product_graph(6, 6, True)
    compare(pkg, g)
    r = mapgen.random_graph(200_000, 1, 6, acc_p, seed=8, variant="plain")
    compare(pkg, r, pkg.MAP_FLAG_FRONTIER_START)


@pytest.mark.parametrize("n,layers,plant", [(2_000_003, 100, True), (3_000_000, 30, True), (2_500_000, 9, False)])
def test_floods(pkg, n, layers, plant):
    """Lists of a large share of the whole graph: into scan mode and back, in one iteration and in several."""
    g = mapgen.layered_graph(n, layers, seed=n, plant=plant, acc_p=0.01 if plant else 0.3)
    compare(pkg, g, pkg.MAP_FLAG_FRONTIER_START, runs=1)
    want = oracle.run_graph(g)
    h = pkg.map_create(g.n, g.rowptr, g.colidx, pkg.pack_bits(g.acc))
    try:  # stopped inside and outside of scan mode, then whole
        for k in (1, 2, 4, 6, 9, 12, 20):
            if k < want.rounds[0]:
                r = pkg.map_run(h, flags=pkg.MAP_FLAG_FRONTIER_START, max_inner=k, allow_limit=True)
                assert r.status == pkg.MAP_ERR_LIMIT and r.rounds == [k]
        r = pkg.map_run(h, flags=pkg.MAP_FLAG_FRONTIER_START)
        assert (r.verdict, r.outer, r.rounds, r.relaxations) == (want.verdict, want.outer, want.rounds, want.relaxations)
    finally:
        pkg.map_destroy(h)


def test_batch_flood(pkg):
    gs = [mapgen.layered_graph(n, max(8, n // 16777), seed=n, plant=bool(i % 2))
          for i, n in enumerate([900_000, 800_000, 300_000, 50_000, 7000, 400_001])]
    h = pkg.map_batch_create([(g.n, g.rowptr, g.colidx, pkg.pack_bits(g.acc)) for g in gs])
    try:
        for sched in (0, 1):
            out = np.empty(sum(g.n for g in gs), np.uint32)
            rs = pkg.map_batch_run(h, len(gs), sched=sched, flags=pkg.MAP_FLAG_FRONTIER_START, map_out=out)
            off = 0
            for g, r in zip(gs, rs):
                want = oracle.run_graph(g)
                assert (r.verdict, r.witness, r.outer) == (want.verdict, want.witness, want.outer)
                assert np.array_equal(out[off:off + g.n], want.map)
                if sched == 0:
                    assert (r.rounds, r.relaxations) == (want.rounds, want.relaxations)
                off += g.n
    finally:
        pkg.map_destroy(h)


LIMIT = 65536  # vertices of the largest graph that is set up in one cluster (131,072 entries)


@pytest.mark.parametrize("n,m", [(1, 0), (1, 3), (33, 0), (1023, 5000), (1025, 1024), (16_385, 65_537),
                                 (LIMIT, 2 * LIMIT), (LIMIT, 2 * LIMIT + 1), (LIMIT + 1, 2 * LIMIT), (700, 2 * LIMIT)])
@pytest.mark.parametrize("where", ["device", "unaligned", "host", "pinned"])
def test_set_up(pkg, n, m, where):
    """Graphs around the limits of the one-cluster set-up, wherever the input lies: rows without entries, repeated
    entries, one row of a quarter of all entries, bits set past the last vertex."""
    rng = np.random.default_rng(n + m)
    at = np.sort(rng.integers(0, n, m))
    at[: m // 4] = at[: max(1, m // 4)][0] if m else 0
    rowptr = np.searchsorted(np.sort(at), np.arange(n + 1)).astype(np.uint32)
    rowptr[n] = m
    col = rng.integers(0, n, m).astype(np.uint32)
    acc = (rng.random(n) < 0.1).astype(np.uint8)
    g = mapgen.Graph(n, rowptr, col, acc, (0,) * 8, "set-up", {})
    want = oracle.run_graph(g)
    bits = pkg.pack_bits(acc).copy()
    if n & 31:
        bits[-1] |= np.uint32(0xFFFFFFFF << (n & 31) & 0xFFFFFFFF)
    args = [rowptr, col, bits]
    if where != "host":
        shift = 1 if where == "unaligned" else 0
        args = [torch.from_numpy(np.concatenate([np.zeros(shift, np.uint32), x]).view(np.int32)) for x in args]
        args = [(x.pin_memory() if where == "pinned" else x.cuda())[shift:] for x in args]
    h = pkg.map_create(n, args[0], args[1] if m else None, args[2])
    try:
        assert pkg.map_graph_info(h) == (n, m)
        for flags in (pkg.MAP_FLAG_FRONTIER_START, pkg.MAP_FLAG_DENSE_START):
            out = torch.empty(n, dtype=torch.int32, device="cuda")
            r = pkg.map_run(h, flags=flags, map_out=out)
            assert (r.verdict, r.witness, r.outer) == (want.verdict, want.witness, want.outer)
            assert (r.rounds, r.relaxations) == (want.rounds, want.relaxations)
            assert np.array_equal(out.cpu().numpy().view(np.uint32), want.map)
        assert np.array_equal(np.asarray(pkg.map_graph_csr(h)[1]).view(np.uint32)[:m], col)
    finally:
        pkg.map_destroy(h)


@pytest.mark.parametrize("n", [40, 20_000, LIMIT])
@pytest.mark.parametrize("fault", ["decreasing", "entry", "first"])
@pytest.mark.parametrize("on_device", [False, True])
def test_set_up_refuses(pkg, n, fault, on_device):
    rowptr = np.arange(n + 1, dtype=np.uint32)
    col = np.arange(n, dtype=np.uint32)
    if fault == "decreasing":
        rowptr[n - 1] = n + 1
    elif fault == "entry":
        col[n // 2] = n
    else:
        col[0] = 0xFFFFFFFF
    args = [rowptr, col, np.zeros((n + 31) // 32, np.uint32)]
    if on_device:
        args = [torch.from_numpy(x.view(np.int32)).cuda() for x in args]
    with pytest.raises(pkg.MapError, match="CSR"):
        pkg.map_create(n, *args)


def test_large_jobs_run_alone(pkg):
    """Queued behind a long job, jobs of up to 65,536 vertices share runs, larger ones run alone."""
    big = mapgen.layered_graph(4_000_000, 240, seed=8)
    gs = [mapgen.layered_graph(LIMIT + d, 12, seed=40 + i, plant=bool(i & 1)) for i, d in enumerate([-1, 0, 1, 0, 1, -7])]
    with pkg.Server(slots=1) as sv:
        first = sv.submit(big.n, big.rowptr, big.colidx, pkg.pack_bits(big.acc))
        ids = [sv.submit(g.n, g.rowptr, g.colidx, pkg.pack_bits(g.acc)) for g in gs]
        left, done = {first, *ids}, {}
        deadline = time.time() + 60
        while left and time.time() < deadline:
            for jid in list(left):
                got = sv.poll(jid)
                if got is not None:
                    done[jid] = got
                    left.discard(jid)
    assert not left
    for g, jid in zip(gs, ids):
        r, mp = done[jid]
        want = oracle.run_graph(g)
        assert (r.verdict, r.witness, r.outer, r.relaxations) == (want.verdict, want.witness, want.outer, want.relaxations)
        assert np.array_equal(mp, want.map)
        assert (r.batch_jobs > 1) == (g.n <= LIMIT), g.n
