"""What one kernel of a whole run leaves to the next (k_run to k_own to k_tail), against the oracle: graphs of a batch that
end in the iteration after which the rest is renumbered, counters that scan mode has used, rows that are
reached in every round, graphs of few vertices and many entries."""
import time

import numpy as np
import pytest

import mapgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

OWN = 152 * 12288  # vertices that k_own holds whole


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__

    __graft_entry__.build()
    import paper_0912_2555_gb300 as p

    return p


def padded(g, n):
    """g with vertices without edges behind it."""
    rowptr = np.concatenate([g.rowptr, np.full(n - g.n, g.rowptr[-1], np.uint32)])
    acc = np.concatenate([g.acc, np.zeros(n - g.n, np.uint8)])
    return mapgen.Graph(n, rowptr, g.colidx, acc, (0,) * 8, g.name, {})


def same(r, want, sched, got):
    assert (r.verdict, r.witness, r.outer) == (want.verdict, want.witness, want.outer)
    assert np.array_equal(got, want.map)
    if sched == 0:
        assert (r.rounds, r.relaxations) == (want.rounds, want.relaxations)


def two_cycles(n):
    """Two accepting vertices on cycles, the smaller one leads to the larger: 5 is the witness, 2 is left with a value."""
    rows = [[] for _ in range(n)]
    rows[2], rows[5] = [2, 5], [5]
    return mapgen.from_lists(rows, [int(v in (2, 5)) for v in range(n)])


@pytest.mark.parametrize("large", [OWN + 1, 3_000_000])
def test_batch_renumbered_while_graphs_end(pkg, large):
    """Small graphs end with a cycle in iteration 1, the large ones go on renumbered: the ended ones stay as they are."""
    gs = [two_cycles(6), padded(mapgen.layered_graph(90_000, 30, seed=7), large), two_cycles(70)]
    gs += [mapgen.tiny_graph(seed, 40, max_deg=3, acc_p=0.4) for seed in range(12)]
    gs += [mapgen.layered_graph(50_000, 20, seed=9), mapgen.layered_graph(5000, 8, seed=10, plant=True)]
    wants = [oracle.run_graph(g) for g in gs]
    assert max(w.outer for w in wants) > 2 and sum(w.verdict == 1 and w.outer == 1 for w in wants) > 4
    h = pkg.map_batch_create([(g.n, g.rowptr, g.colidx, pkg.pack_bits(g.acc)) for g in gs])
    try:
        for sched in (0, 1):
            out = np.empty(sum(g.n for g in gs), np.uint32)
            rs = pkg.map_batch_run(h, len(gs), sched=sched, flags=pkg.MAP_FLAG_FRONTIER_START, map_out=out)
            off = 0
            for g, r, want in zip(gs, rs, wants):
                same(r, want, sched, out[off:off + g.n])
                off += g.n
    finally:
        pkg.map_destroy(h)


def test_served_batch_on_a_share_of_the_chip(pkg):
    """The same through a server: a worker's share of the chip holds fewer vertices, so that a shared run of a few hundred
    thousand is renumbered."""
    n = 65_536
    gs = [padded(mapgen.layered_graph(12_000, 14, seed=s), n) for s in range(6)]
    gs += [two_cycles(n), two_cycles(6), padded(mapgen.layered_graph(4000, 8, seed=4, plant=True), n)]
    wants = [oracle.run_graph(g) for g in gs]
    length = n + 1  # a chain: one vertex per round, so that every worker is busy while the jobs are queued
    chain = mapgen.Graph(length, np.concatenate([[0], np.arange(length)]).astype(np.uint32), np.arange(length - 1, dtype=np.uint32),
                         (np.arange(length) == 0).astype(np.uint8), (0,) * 8, "chain", {})
    with pkg.Server(slots=8) as sv:
        first = [sv.submit(chain.n, chain.rowptr, chain.colidx, pkg.pack_bits(chain.acc)) for _ in range(8)]
        for sched in (0, 1):
            ids = [sv.submit(g.n, g.rowptr, g.colidx, pkg.pack_bits(g.acc), sched=sched) for g in gs]
            left, done = set(ids), {}
            deadline = time.time() + 60
            while left and time.time() < deadline:
                for jid in list(left):
                    got = sv.poll(jid)
                    if got is not None:
                        done[jid] = got
                        left.discard(jid)
            assert not left
            assert sched or max(r.batch_jobs for r, _ in done.values()) == len(gs)
            for want, jid in zip(wants, ids):
                r, mp = done[jid]
                assert (r.verdict, r.witness, r.outer) == (want.verdict, want.witness, want.outer)
                assert sched or r.relaxations == want.relaxations
                assert np.array_equal(mp, want.map)
        for jid in first:
            while sv.poll(jid) is None:
                pass


@pytest.mark.parametrize("n", [OWN + 1000, 4_000_000])
def test_scan_mode_then_the_grid_kernel(pkg, n):
    """Accepting h1 > h2 > h3 and h0.  The same quarter of the rows holds h1 and h2 (their iterations end in scan mode), 20,000
    of these hold h3 (renumbered, the rest in k_own), none holds h0: the fourth iteration gives nobody a value and is
    the last."""
    rows = n // 4
    deg = np.zeros(n, np.int64)
    deg[:rows] = 2
    deg[:20_000] = 3
    rowptr = np.zeros(n + 1, np.uint32)
    np.cumsum(deg, out=rowptr[1:])
    col = np.tile(np.array([n - 1, n - 2], np.uint32), rows + 10_000)
    col[rowptr[:rows]], col[rowptr[:rows] + 1] = n - 1, n - 2
    col[rowptr[:20_000] + 2] = n - 3
    acc = np.zeros(n, np.uint8)
    acc[n - 4:] = 1
    g = mapgen.Graph(n, rowptr, col[:rowptr[-1]], acc, (0,) * 8, "stars", {})
    want = oracle.run_graph(g)
    assert want.outer == 4
    h = pkg.map_create(g.n, g.rowptr, g.colidx, pkg.pack_bits(g.acc))
    try:
        for sched in (0, 1):
            for kw in ({}, dict(max_outer=want.outer)):
                out = np.empty(n, np.uint32)
                r = pkg.map_run(h, sched=sched, flags=pkg.MAP_FLAG_FRONTIER_START, map_out=out, **kw)
                same(r, want, sched, out)
                assert (r.edges_total, r.accepting_left) == (4 * g.m, 1)
    finally:
        pkg.map_destroy(h)


@pytest.mark.parametrize("n", [60_000, OWN - 40, OWN + 100_000])
def test_batched_rows_reached_in_every_round(pkg, n):
    """One value runs down a chain of 200 vertices, and thousands of rows in one block's share hold the whole chain: they are
    in every round's frontier, and each time their length belongs to the relaxation count of an asynchronous batch too, also
    where the next round's pushes come in before their block has looked."""
    length = 200
    share = np.arange(n) // 32 % 152 == 0
    wides = np.flatnonzero(share)[:10_000]
    chain = np.random.default_rng(5).permutation(np.flatnonzero(~share))[:length]
    deg = np.zeros(n, np.int64)
    deg[wides], deg[chain[1:]] = length - 1, 1
    rowptr = np.zeros(n + 1, np.uint32)
    np.cumsum(deg, out=rowptr[1:])
    col = np.zeros(int(rowptr[-1]), np.uint32)
    col[(rowptr[wides][:, None] + np.arange(length - 1)).ravel()] = np.tile(chain[1:], wides.size)
    col[rowptr[chain[1:]]] = chain[:-1]
    acc = np.zeros(n, np.uint8)
    acc[chain[0]] = 1
    g = mapgen.Graph(n, rowptr, col, acc, (0,) * 8, "chain", {})
    small = mapgen.tiny_graph(3, 20)
    h = pkg.map_batch_create([(x.n, x.rowptr, x.colidx, pkg.pack_bits(x.acc)) for x in (g, small)])
    try:
        for sched in (1, 0, 1):
            r = pkg.map_batch_run(h, 2, sched=sched, flags=pkg.MAP_FLAG_FRONTIER_START)[0]
            assert (r.verdict, r.outer) == (0, 1)
            # the whole chain but its head pushes to them, from round 2 to the last; a chain vertex once, from round 2 on
            assert r.relaxations == g.m + (r.inner_iters - 1) * wides.size * (length - 1) + length - 2, sched
    finally:
        pkg.map_destroy(h)


TAIL_N, TAIL_M = 16384, 262144  # the largest graph that runs in one cluster


def clumps(n, m, seed):
    """m entries, each row's among its next vertices: reader lists as long as rows, no cycle but through the last rows."""
    rng = np.random.default_rng(seed)
    row = np.sort(rng.integers(0, n, m))
    rowptr = np.searchsorted(row, np.arange(n + 1)).astype(np.uint32)
    col = np.minimum(row + 1 + (rng.random(m) * max(1, n // 20)).astype(np.int64), n - 1).astype(np.uint32)
    acc = (rng.random(n) < 0.02).astype(np.uint8)
    acc[n - 1] = 0
    return mapgen.Graph(n, rowptr, col, acc, (0,) * 8, "clumps", {})


@pytest.mark.parametrize("n,m,launches", [(TAIL_N, TAIL_M, 1), (TAIL_N, TAIL_M + 1, 2), (700, TAIL_M, 1), (700, TAIL_M + 1, 2),
                                          (5000, 1_000_000, 2)])
def test_graphs_of_many_entries_use_the_whole_chip(pkg, n, m, launches):
    """Sixteen SMs fall behind the whole chip where every vertex has many readers, however few the vertices."""
    g = clumps(n, m, n)
    want = oracle.run_graph(g, max_outer=12)
    h = pkg.map_create(g.n, g.rowptr, g.colidx, pkg.pack_bits(g.acc))
    try:
        for sched in (0, 1):
            out = np.empty(n, np.uint32)
            r = pkg.map_run(h, sched=sched, map_out=out, max_outer=12, allow_limit=True)
            same(r, want, sched, out)
            assert r.launches == launches
    finally:
        pkg.map_destroy(h)


@pytest.mark.parametrize("pad", [100_000, OWN])
def test_renumbered_graph_of_many_entries(pkg, pad):
    """A graph of few vertices and many entries inside a large one: what is left after an iteration is small enough for the
    cluster by its vertices and too large by its entries, later by neither."""
    core = clumps(6000, 400_000, 3)
    g = padded(core, core.n + pad)
    want = oracle.run_graph(g)
    assert want.outer > 20
    h = pkg.map_create(g.n, g.rowptr, g.colidx, pkg.pack_bits(g.acc))
    try:
        for sched in (0, 1):
            out = np.empty(g.n, np.uint32)
            r = pkg.map_run(h, sched=sched, flags=pkg.MAP_FLAG_FRONTIER_START, map_out=out)
            same(r, want, sched, out)
    finally:
        pkg.map_destroy(h)


@pytest.mark.parametrize("n,m,launches", [(TAIL_N, 300_000, 2), (TAIL_N + 1, 60_000, 3), (40_001, 500_000, 3), (65_536, 524_288, 3)])
@pytest.mark.parametrize("on_device", [False, True])
def test_static_runs_over_the_grid(pkg, n, m, launches, on_device):
    """map_run_static: set-up in one cluster, runs of more than 16,384 vertices over the grid, what is left of them in the
    cluster; an invalid graph is still refused, and the call after that one sees nothing of either."""
    gs = [clumps(n, m, n), mapgen.layered_graph(n, max(8, n // 4000), seed=n)]
    for g in gs * 2:
        want = oracle.run_graph(g, max_outer=12)
        args = [g.rowptr, g.colidx, pkg.pack_bits(g.acc)]
        if on_device:
            args = [torch.from_numpy(x.view(np.int32)).cuda() for x in args]
        for sched in (0, 1):
            out = np.full(n, 7, np.uint32)
            r = pkg.map_run_static(n, *args, sched=sched, map_out=out, max_outer=12, allow_limit=True)
            same(r, want, sched, out)
            assert r.launches == launches
            bad = [args[0], args[1].copy() if not on_device else args[1].clone(), args[2]]
            bad[1][g.m // 2] = n
            with pytest.raises(pkg.MapError, match="CSR"):
                pkg.map_run_static(n, *bad, sched=sched, map_out=out)
