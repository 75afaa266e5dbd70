"""Scan mode of whole runs (lists of a large share of a graph above k_own's capacity): every block adds up the hits of
several chunks and pushes them once the next chunk might not fit, a decision that all its warps must take alike."""
import os
import re

import numpy as np
import pytest

import mapgen
import oracle

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0912_2555_gb300", "csrc")


def test_the_hit_count_is_read_between_two_block_barriers():
    """The shared count of scan_round is read after a block barrier, and another one follows before the branch on it: else a
    fast warp adds the next chunk's hits while a slow one still reads, and the warps part ways inside a block barrier."""
    with open(os.path.join(CSRC, "map_run.cuh")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    body = text[text.index("bool scan_round("):text.index("bool leave_scan(")]
    reads = list(re.finditer(r"__syncthreads\(\);\s*const uint32_t nq = sh\.ln;(.*?)if \(nq", body, re.S))
    assert len(reads) == len(re.findall(r"= sh\.ln;", body)) == 1
    assert reads[0].group(1).strip() == "__syncthreads();"


def stars(n, share, hubs=64):
    """`hubs` accepting vertices at the top; a share of the others reads one of them each, and a tenth of those is read on."""
    rng = np.random.default_rng(int(n * share))
    inner = n - hubs
    reads = rng.random(inner) < share
    on = (rng.random(inner) < 0.1) & ~reads
    deg = np.zeros(n, np.int64)
    deg[:inner] = reads | on
    rowptr = np.zeros(n + 1, np.uint32)
    np.cumsum(deg, out=rowptr[1:])
    to = rng.integers(inner, n, inner)
    to[on] = rng.choice(np.flatnonzero(reads), int(on.sum()))
    acc = np.zeros(n, np.uint8)
    acc[inner:] = 1
    return mapgen.Graph(n, rowptr, to[reads | on].astype(np.uint32), acc, (0,) * 8, "stars", {})


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1_900_003, 5_000_011])
@pytest.mark.parametrize("share", [0.07, 0.32, 0.48, 0.5, 0.52, 0.9])
def test_hits_around_the_room_for_another_chunk(n, share):
    """Chunks of 2,048 vertices with hits from a few to nearly all of them: at a half two chunks just fill the staged list."""
    torch = pytest.importorskip("torch")
    import __graft_entry__

    __graft_entry__.build()
    import paper_0912_2555_gb300 as pkg

    g = stars(n, share)
    want = oracle.run_graph(g)
    h = pkg.map_create(g.n, g.rowptr, g.colidx, pkg.pack_bits(g.acc))
    b = pkg.map_batch_create([(g.n, g.rowptr, g.colidx, pkg.pack_bits(g.acc))] * 2)
    try:
        out = torch.empty(3 * n, dtype=torch.int32, device="cuda")
        for sched in (0, 1, 0, 1):
            rs = pkg.map_batch_run(b, 2, sched=sched, flags=pkg.MAP_FLAG_FRONTIER_START, map_out=out[:2 * n])
            rs.append(pkg.map_run(h, sched=sched, flags=pkg.MAP_FLAG_FRONTIER_START, map_out=out[2 * n:]))
            for r, got in zip(rs, out.cpu().numpy().view(np.uint32).reshape(3, n)):
                assert (r.verdict, r.witness, r.outer) == (want.verdict, want.witness, want.outer)
                if sched == 0:
                    assert (r.rounds, r.relaxations) == (want.rounds, want.relaxations)
                assert np.array_equal(got, want.map)
    finally:
        pkg.map_destroy(h)
        pkg.map_destroy(b)
