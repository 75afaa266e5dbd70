"""Asynchronous floods: a vertex whose value rises again before it is pushed is pushed once, with the value it has by then.
The relaxations say how much was pushed for nothing."""
import numpy as np
import pytest

import mapgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__

    __graft_entry__.build()
    import paper_0912_2555_gb300 as p

    return p


def waves(n, deg):
    """Every row holds `deg` vertices of the next n / 40: values move down in waves, the larger ones behind the smaller."""
    rng = np.random.default_rng(n)
    v = np.repeat(np.arange(n), deg)
    col = np.minimum(v + 1 + (rng.random(v.size) * (n // 40)).astype(np.int64), n - 1).astype(np.uint32)
    acc = (rng.random(n) < 0.01).astype(np.uint8)
    acc[n - 1] = 0
    return mapgen.Graph(n, (np.arange(n + 1) * deg).astype(np.uint32), col, acc, (0,) * 8, "waves", {})


# pushes per edge and iteration: the dense start takes 6.8 and 4.7 on such graphs of 10^6 and 4 * 10^6 vertices, pushing
# what a vertex had when it was found took 18 and 17
@pytest.mark.parametrize("n,deg,most", [(1_000_000, 16, 11), (4_000_000, 16, 13)])
def test_pushes_per_edge(pkg, n, deg, most):
    g = waves(n, deg)
    h = pkg.map_create(g.n, g.rowptr, g.colidx, pkg.pack_bits(g.acc))
    try:
        out, want = np.empty(n, np.uint32), np.empty(n, np.uint32)
        # (a graph of this size takes the oracle a minute; the synchronous dense start is compared with it elsewhere)
        pkg.map_run(h, sched=0, flags=pkg.MAP_FLAG_DENSE_START, max_outer=3, map_out=want, allow_limit=True)
        for _ in range(2):
            r = pkg.map_run(h, sched=1, flags=pkg.MAP_FLAG_FRONTIER_START, max_outer=3, map_out=out, allow_limit=True)
            assert r.outer == 3 and np.array_equal(out, want)
            assert r.relaxations <= most * 3 * g.m, r.relaxations / (3 * g.m)
    finally:
        pkg.map_destroy(h)
