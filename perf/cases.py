"""Performance cases of the library: what a verification program has it do, through its Python API.

A case names a graph family, a size, a schedule and the way the library is called:

  static    map_run_static: one call on a small graph, inputs and map on the device
  resident  map_run on a graph that was created before (a handle kept between runs)
  check     Graph(...), run, close: one verdict for a graph seen for the first time
  lasso     map_run on a kept graph, then the counterexample for its cycle verdict
  batch     map_batch_run on a kept batch of uneven graphs, 40 % with a planted accepting cycle
  serve     a burst of uneven jobs submitted to a kept Server and polled to the last result

Graph families, made on the GPU from the seed (integer structure, no file):

  random    out-degree 1 to 6, uniform targets, 3 % accepting; accepting vertices on the acyclic
            part, or (cycle) with a 20-vertex cycle closed through the largest of them
  layered   consecutive layers, geometric out-degree with mean 4, 92 % of the edges into the next
            layer and the others back over up to 50 layers, 1 % accepting on no cycle; or (cycle)
            with one edge that closes a cycle
  product   k cyclic s-state processes times a two-state automaton; a process may advance when its
            right neighbour is an even number of steps from where it began; in lock-step (one
            successor per state) or interleaved (one process moves per step)
"""
import math

import numpy as np
import torch

import paper_0912_2555_gb300 as pkg

SYNC, ASYNC = pkg.MAP_SCHED_SYNC, pkg.MAP_SCHED_ASYNC


def listed():
    return [
        # a small model checked inside a loop that may not allocate: launches and waits
        dict(name="static-1k-sync", how="static", family="random", n=1000, cycle=False, sched="sync"),
        # the 16,384-vertex random graph kept and run again: latency of a small run, canonical counts
        dict(name="resident-16k-sync", how="resident", family="random", n=16384, cycle=False, sched="sync"),
        # a small graph seen once (with a cycle): create, run and destroy from device arrays
        dict(name="check-16k-async", how="check", family="random", n=16384, cycle=True, sched="async", source="device"),
        # an ordinary model of a million states, odd size
        dict(name="resident-1M-async", how="resident", family="layered", n=1000003, cycle=False, sched="async"),
        # a large model with the canonical round and relaxation counts
        dict(name="resident-16M-sync", how="resident", family="layered", n=1 << 24, cycle=False, sched="sync"),
        # the largest: 2^26 states in 4,000 layers, as the benchmark runs it
        dict(name="resident-64M-async", how="resident", family="layered", n=1 << 26, cycle=False, sched="async"),
        # a deterministic system: every state has one successor
        dict(name="product-8x7-async", how="resident", family="product", k=8, s=7, interleave=False, sched="async"),
        # an interleaved process product: many rounds over lists of all sizes, many accepting states
        dict(name="product-i-7x7-sync", how="resident", family="product", k=7, s=7, interleave=True, sched="sync"),
        # one verdict end to end from page-locked host arrays, the map copied back to the host
        dict(name="check-4M-async", how="check", family="layered", n=4000037, cycle=False, sched="async", source="host"),
        # a graph with a cycle, and the counterexample that shows it from the initial state
        dict(name="lasso-1M-async", how="lasso", family="random", n=1000003, cycle=True, sched="async"),
        # many uneven graphs in one run
        dict(name="batch-64-sync", how="batch", count=64, lo=1000, hi=1000000, sched="sync"),
        # jobs that arrive together, median 10^5 states, half of them deterministic products
        dict(name="serve-32-async", how="serve", count=32, median=100000, hi=2000000, sched="async"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    how = rng.choice(["static", "resident", "resident", "resident", "check", "check", "lasso", "batch", "serve"])
    sched = rng.choice(["sync", "async"])
    if how == "batch":
        return dict(how=how, count=rng.randint(2, 96), lo=1000, hi=_log_int(rng, 10000, 1000000), sched=sched)
    if how == "serve":
        return dict(how=how, count=rng.randint(4, 40), median=_log_int(rng, 10000, 200000), hi=2000000, sched=sched)
    if how == "lasso":
        return dict(how=how, family="random", n=_log_int(rng, 1000, 1000000), cycle=True, sched=sched)
    if how == "static":
        family = rng.choice(["random", "layered"])
        return dict(how=how, family=family, n=_log_int(rng, 300, 60000), cycle=rng.random() < 0.5, sched=sched)
    family = rng.choice(["random", "layered", "layered", "product"])
    if family == "product":
        interleave = rng.random() < 0.5
        c = dict(family=family, k=rng.randint(4, 7), s=rng.randint(5, 7), interleave=interleave, sched=sched)
    else:
        top = 1 << 25 if family == "layered" else 1 << 20
        c = dict(family=family, n=_log_int(rng, 1000, top if how == "resident" else top // 4),
                 cycle=rng.random() < 0.3, sched=sched)
    if how == "check":
        return dict(c, how=how, source=rng.choice(["device", "host"]))
    # the start of every outer iteration may be asked for, or be left to the library
    return dict(c, how=how, start=rng.choice(["default", "default", "dense", "frontier"]))


# ------------------------------------------------------------------ graphs --

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _rand(count, gen):
    return torch.rand(count, generator=gen, device="cuda", dtype=torch.float64)


def _pick(lo, hi, gen):
    """A uniform integer in [lo, hi) for each pair (lo when the range is empty)."""
    return lo + (_rand(lo.numel(), gen) * (hi - lo)).long().minimum((hi - lo - 1).clamp(min=0))


def _random(n, cycle, seed):
    gen = _gen(seed)
    dag = max(2, n // 12)  # vertices [0, dag) lead to larger ids only, a third of their edges to each other
    deg = torch.randint(1, 7, (n,), generator=gen, device="cuda")
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = deg.cumsum(0)
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
    near = (row < dag - 1) & (_rand(row.numel(), gen) < 1 / 3)
    lo = torch.where(near, row + 1, torch.full_like(row, dag))
    col = _pick(lo, torch.where(near, torch.full_like(row, dag), torch.full_like(row, n)), gen)
    acc = torch.zeros(n, dtype=torch.bool, device="cuda")
    acc[torch.randperm(dag, generator=gen, device="cuda")[: max(1, int(0.03 * n))]] = True
    if cycle:  # 20 vertices in a ring through the largest accepting one: the first entry of each row
        top = int(acc.nonzero().max())
        ring = torch.randperm(n - dag, generator=gen, device="cuda")[: min(19, n - dag)] + dag
        ring = torch.cat([torch.tensor([top], device="cuda"), ring])
        col[rowptr[ring]] = ring.roll(-1)
    return rowptr, col, acc


def _layered(n, cycle, seed, window=50, segment=16):
    gen = _gen(seed)
    layers = max(8, round(n / 16777))
    ids = torch.arange(n, device="cuda")
    acc = _rand(n, gen) < 0.01
    start = (torch.arange(layers + 1, device="cuda") * n + layers - 1) // layers
    alist, nlist = ids[acc], ids[~acc]
    aoff, noff = torch.searchsorted(alist, start), torch.searchsorted(nlist, start)
    deg = (1 + (_rand(n, gen).clamp_(min=1e-300).log_() / math.log(0.75)).floor_()).clamp_(max=64).long()
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = deg.cumsum(0)
    col = torch.empty(int(rowptr[-1]), dtype=torch.int32, device="cuda")
    step = 1 << 23
    for v0 in range(0, n, step):
        v1 = min(n, v0 + step)
        row = torch.repeat_interleave(ids[v0:v1], deg[v0:v1])
        lay = row * layers // n
        nxt, after = (lay + 1).clamp(max=layers), (lay + 2).clamp(max=layers)
        fwd = (lay + 1 < layers) & ((lay == 0) | (_rand(row.numel(), gen) < 0.92))
        to_acc = fwd & acc[row] & ((lay + 1) % segment != 0) & (aoff[after] > aoff[nxt]) & (_rand(row.numel(), gen) < 0.5)
        lo = torch.where(to_acc, aoff[nxt], torch.where(fwd, noff[nxt], noff[(lay - window).clamp(min=0)]))
        hi = torch.where(to_acc, aoff[after], torch.where(fwd, noff[after], noff[lay]))
        at = _pick(lo, hi, gen)
        to = nlist[at.clamp(max=max(0, nlist.numel() - 1))]
        if alist.numel():
            to = torch.where(to_acc, alist[at.clamp(max=alist.numel() - 1)], to)
        col[int(rowptr[v0]):int(rowptr[v1])] = to.int()
    if cycle and alist.numel():  # an accepting vertex a with a non-accepting successor w: w's first entry becomes a
        for a in alist[torch.randperm(alist.numel(), generator=gen, device="cuda")[:64]].tolist():
            to = col[int(rowptr[a]):int(rowptr[a + 1])].long()
            to = to[~acc[to]]
            if to.numel():
                col[int(rowptr[int(to[0])])] = a
                break
    return rowptr, col, acc


def _product(k, s, interleave, seed):
    rng = np.random.default_rng(int(seed) + 1000003 * k + 31 * s)
    # where each process begins, and the local state of process 0 that the automaton accepts on
    begin, mark = [int(v) for v in rng.integers(0, s, k)], int(rng.integers(0, s))
    total = s ** k
    ids = torch.arange(total, device="cuda")
    x = [(ids // s ** i) % s for i in range(k)]
    may = [(x[(i + 1) % k] - begin[(i + 1) % k]) % s % 2 == 0 for i in range(k)]
    if not interleave:
        y = [torch.where(may[i], (x[i] + 1) % s, x[i]) for i in range(k)]
        to = sum(y[i] * s ** i for i in range(k)) + (y[0] == mark).long() * total
        deg = torch.ones(total, dtype=torch.int64, device="cuda")
    else:
        opts = []
        for i in range(k):
            xi = (x[i] + 1) % s
            y0 = xi if i == 0 else x[0]
            opts.append(torch.where(may[i], ids + (xi - x[i]) * s ** i + (y0 == mark).long() * total, -1))
        stuck = ~torch.stack(may).any(0)  # no process can move: a stutter step
        opts.append(torch.where(stuck, ids + (x[0] == mark).long() * total, -1))
        grid = torch.stack(opts, 1)
        deg = (grid >= 0).sum(1)
        to = grid[grid >= 0]
    rowptr = torch.zeros(2 * total + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = torch.cat([deg, deg]).cumsum(0)
    return rowptr, torch.cat([to, to]), ids.new_zeros(2 * total).bool().index_fill_(0, ids + total, True)


def _graph(c, seed):
    """(rowptr, colidx, accepting flags) of the case's graph, on the device."""
    if c["family"] == "random":
        return _random(c["n"], c["cycle"], seed)
    if c["family"] == "layered":
        return _layered(c["n"], c["cycle"], seed)
    return _product(c["k"], c["s"], c["interleave"], seed)


def _members(c):
    """The graphs of a batch (sizes log-uniform) or of a burst of jobs (sizes lognormal): the same
    sizes for every seed of a case."""
    rng = np.random.default_rng([c["count"], c["hi"]])
    if c["how"] == "batch":
        n = np.exp(rng.uniform(math.log(c["lo"]), math.log(c["hi"]), c["count"])).astype(int)
        plant = rng.permutation(c["count"]) < round(0.4 * c["count"])
        return [dict(family="layered", n=int(n[i]), cycle=bool(plant[i])) for i in range(c["count"])]
    out = []
    for size in np.clip(c["median"] * np.exp(1.5 * rng.standard_normal(c["count"])), 1000, c["hi"]):
        if rng.random() < 0.5:
            out.append(dict(family="layered", n=int(size), cycle=False))
        else:  # the product of 5- to 7-state processes nearest to the size
            s = int(rng.integers(5, 8))
            out.append(dict(family="product", k=max(4, round(math.log(size / 2) / math.log(s))), s=s, interleave=False))
    return out


def _packed(acc):
    """The accepting set as the library takes it: one bit per vertex, least significant first."""
    bits = torch.zeros((acc.numel() + 31) // 32 * 32, dtype=torch.int64, device="cuda")
    bits[: acc.numel()] = acc.long()
    words = (bits.view(-1, 32) << torch.arange(32, device="cuda")).sum(1)
    return torch.where(words >= 1 << 31, words - (1 << 32), words).int()


def _arrays(c, seed):
    rowptr, col, acc = _graph(c, seed)
    return rowptr.int(), col.int().contiguous(), _packed(acc)


# ----------------------------------------------------------- prepare, run --

class _Batch:
    """A batch handle, destroyed with its owner."""

    def __init__(self, graphs):
        self.handle = pkg.map_batch_create(graphs)

    def __del__(self):
        pkg.map_destroy(self.handle)


def prepare(case, seed):
    st = dict(case, sched=SYNC if case["sched"] == "sync" else ASYNC)
    how = case["how"]
    if how in ("batch", "serve"):
        members = [(int(rp.numel()) - 1, rp, ci, ab) for rp, ci, ab in
                   (_arrays(m, seed * 1009 + i) for i, m in enumerate(_members(case)))]
        if how == "batch":
            st["batch"] = _Batch(members)
            st["out"] = torch.empty(sum(g[0] for g in members), dtype=torch.int32, device="cuda")
        else:
            host = lambda t: t.cpu().numpy().view(np.uint32)  # noqa: E731
            st["jobs"] = [(n, host(rp), host(ci), host(ab)) for n, rp, ci, ab in members]
            st["server"] = pkg.Server(hbm_budget_bytes=2 << 30, slots=8)
        return st
    rp, ci, ab = _arrays(case, seed)
    st["n"] = int(rp.numel()) - 1
    st["flags"] = {"default": 0, "dense": pkg.MAP_FLAG_DENSE_START,
                   "frontier": pkg.MAP_FLAG_FRONTIER_START}[case.get("start", "default")]
    if how in ("resident", "lasso"):
        st["graph"] = pkg.Graph(st["n"], rp, ci, acc_bits=ab)
        st["out"] = torch.empty(st["n"], dtype=torch.int32, device="cuda")
    elif case.get("source") == "host":
        st["in"] = tuple(t.cpu().pin_memory() for t in (rp, ci, ab))
        st["out"] = torch.empty(st["n"], dtype=torch.int32).pin_memory()
    else:
        st["in"] = (rp, ci, ab)
        st["out"] = torch.empty(st["n"], dtype=torch.int32, device="cuda")
    return st


def _table(rounds):
    """The rounds of each outer iteration in a table of one size, whatever the graph."""
    return np.array((list(rounds) + [0] * 512)[:512], dtype=np.int64)


def _answer(r, sched, **more):
    """The verdict and what the run says of itself, under the synchronous schedule the canonical counts too."""
    out = dict(verdict=int(r.verdict), witness=int(r.witness), outer=int(r.outer), left=int(r.accepting_left),
               edges=int(r.edges_total), **more)
    if sched == SYNC:
        out.update(rounds=_table(r.rounds), relaxations=int(r.relaxations))
    return out


def _answers(rs, sched):
    """The same for the graphs of a batch or a burst."""
    out = dict(verdict=np.array([r.verdict for r in rs]), witness=np.array([r.witness for r in rs]),
               outer=np.array([r.outer for r in rs]), left=np.array([r.accepting_left for r in rs]),
               edges=np.array([r.edges_total for r in rs]))
    if sched == SYNC:
        out.update(inner=np.array([r.inner_iters for r in rs]), relaxations=np.array([r.relaxations for r in rs]))
    return out


def run(st):
    how, sched = st["how"], st["sched"]
    if how == "static":
        r = pkg.map_run_static(st["n"], *st["in"], sched=sched, map_out=st["out"])
        return _answer(r, sched, map=st["out"])
    if how == "resident":
        r = st["graph"].run(sched=sched, flags=st["flags"], map_out=st["out"])
        return _answer(r, sched, map=st["out"])
    if how == "check":
        rp, ci, ab = st["in"]
        with pkg.Graph(st["n"], rp, ci, acc_bits=ab) as g:
            r = g.run(sched=sched, map_out=st["out"])
        return _answer(r, sched, map=st["out"])
    if how == "lasso":
        r = st["graph"].run(sched=sched, map_out=st["out"])
        prefix, cycle = st["graph"].lasso(r.witness, init=0) if r.verdict else ([], [])
        # (shortest paths are not unique, their lengths are)
        return _answer(r, sched, map=st["out"], prefix=len(prefix), cycle=len(cycle))
    if how == "batch":
        rs = pkg.map_batch_run(st["batch"].handle, st["count"], sched=sched, map_out=st["out"])
        return dict(_answers(rs, sched), map=st["out"])
    waiting = {st["server"].submit(*job, sched=sched): i for i, job in enumerate(st["jobs"])}
    done = [None] * len(st["jobs"])
    while waiting:
        for job in list(waiting):
            got = st["server"].poll(job)
            if got is not None:
                done[waiting.pop(job)] = got
    return dict(_answers([r for r, _ in done], sched), maps=[m.view(np.int32) for _, m in done])


# -------------------------------------------------------------- work, exact --

def _size(c):
    """(vertices, edges) of the case's graph, as its recipe gives them on average."""
    if c["family"] == "random":
        return c["n"], 3.5 * c["n"]
    if c["family"] == "layered":
        return c["n"], 4.0 * c["n"]
    n = 2 * c["s"] ** c["k"]
    return n, n * (c["k"] * ((c["s"] + 1) // 2) / c["s"] if c["interleave"] else 1.0)


def work(case):
    """The matrix and the accepting set read once, the map written once."""
    if case["how"] in ("batch", "serve"):
        sizes = [_size(m) for m in _members(case)]
    else:
        sizes = [_size(case)]
    return {"bytes": float(sum(4 * (n + 1) + 4 * m + n / 8 + 4 * n for n, m in sizes)), "flops": 0.0}


def _distances(n, row, col, source):
    """Edges of a shortest path from `source` along rows to every vertex (-1: none, by at least one edge)."""
    dist = torch.full((n,), -1, dtype=torch.int64, device=row.device)
    front = torch.zeros(n, dtype=torch.bool, device=row.device)
    front[source] = True
    level = 0
    while bool(front.any()):
        level += 1
        new = torch.zeros_like(front)
        new[col[front[row]]] = True
        new &= dist < 0
        dist[new] = level
        front = new
    return dist


def _map(rowptr, col, acc):
    """MAP as it is defined, in synchronous rounds: (verdict, witness, outer, rounds, relaxations, map,
    accepting vertices left)."""
    n, dev = acc.numel(), col.device
    length = rowptr[1:] - rowptr[:-1]
    row = torch.repeat_interleave(torch.arange(n, device=dev), length)
    own = torch.arange(1, n + 1, device=dev)
    acc = acc.clone()
    value = torch.zeros(n, dtype=torch.int64, device=dev)
    rounds, relax = [], 0
    while bool(acc.any()):
        value = torch.zeros(n, dtype=torch.int64, device=dev)
        base = own * acc
        k, frontier = 0, None
        while True:
            k += 1
            relax += col.numel() if frontier is None else int(length[frontier].sum())
            new = value.scatter_reduce(0, row, torch.maximum(base, value)[col], "amax")
            changed = new != value
            value = new
            if not bool(changed.any()):
                break
            frontier = torch.zeros(n, dtype=torch.bool, device=dev)
            frontier[row[changed[col]]] = True
        rounds.append(k)
        on = (value == own).nonzero()
        if on.numel():
            return 1, int(on.min()), len(rounds), rounds, relax, value, int(acc.sum())
        seen = value[value > 0]
        if not seen.numel():
            break
        acc[seen - 1] = False
    return 0, pkg.MAP_NONE, len(rounds), rounds, relax, value, int(acc.sum())


def exact(case, seed):
    sync = case["sched"] == "sync"
    if case["how"] in ("batch", "serve"):
        graphs = [_graph(m, seed * 1009 + i) for i, m in enumerate(_members(case))]
        got = [_map(rp, ci.long(), acc) for rp, ci, acc in graphs]
        maps = [(g[5] - 1).int() for g in got]
        out = dict(verdict=np.array([g[0] for g in got]), witness=np.array([g[1] for g in got]),
                   outer=np.array([g[2] for g in got]), left=np.array([g[6] for g in got]),
                   edges=np.array([g[2] * x[1].numel() for g, x in zip(got, graphs)]))
        if sync:
            out.update(inner=np.array([sum(g[3]) for g in got]), relaxations=np.array([g[4] for g in got]))
        out.update(dict(map=torch.cat(maps)) if case["how"] == "batch" else dict(maps=maps))
        return out
    rowptr, col, acc = _graph(case, seed)
    col = col.long()
    verdict, witness, outer, rounds, relax, value, left = _map(rowptr, col, acc)
    out = dict(verdict=verdict, witness=witness, outer=outer, left=left, edges=outer * col.numel(),
               map=(value - 1).int())
    if sync:
        out.update(rounds=_table(rounds), relaxations=relax)
    if case["how"] == "lasso":
        out.update(prefix=0, cycle=0)
        if verdict:
            row = torch.repeat_interleave(torch.arange(acc.numel(), device=col.device), rowptr[1:] - rowptr[:-1])
            # the prefix without the witness, and the cycle with the witness at both ends
            out.update(prefix=int(_distances(acc.numel(), row, col, 0)[witness]) if witness else 0,
                       cycle=int(_distances(acc.numel(), row, col, witness)[witness]) + 1)
    return out
