"""The work that users of this library have it do, as cases that can be timed.

Every case goes through the public entry points of ``paper_1610_08128_gb300.rcm``. The patterns have
the shapes of the bench's workloads: permuted 2D and 3D grids, nearest-neighbour meshes, a mesh cut
into strips, a scale-free graph, batches and served mixes of grids and meshes. They are built on the
GPU (the package's own generators build the same shapes on the host, which takes minutes at these
sizes); ids are permuted uniformly from the seed, so that no case gains from a natural numbering.

Case fields: ``entry`` is the call (order, noalloc, host, batch, plan, serve, bandwidth), ``shape``
the pattern and the other fields its sizes; ``options`` names what an order call asks for
(default, l2_window, components_first, stored_order); ``shuffled`` stores each row's entries in
random order instead of by column.
"""
import math

import torch

from paper_1610_08128_gb300 import rcm

KNN_DEGREE = {2: 2.73, 3: 3.96}  # mean row length of the symmetrised k-nearest-neighbour meshes


def listed():
    return [
        # one small mesh block, the size a solver asks for again and again: latency of the call
        dict(name="grid2d_64", entry="order", shape="grid", a=64, b=64, c=1, options="default", shuffled=False),
        # the smallest served mesh: a handful of components, a thousand vertices
        dict(name="mesh_1k", entry="order", shape="knn", n=1000, k=3, options="default", shuffled=False),
        # a mid-size 3D block ordered inside a loop that may not allocate
        dict(name="noalloc_30k", entry="noalloc", shape="grid", a=31, b=30, c=32, shuffled=True),
        # a long 2D problem: two thousand narrow levels per sweep
        dict(name="grid2d_1000", entry="order", shape="grid", a=1000, b=1000, c=1, options="default", shuffled=False),
        # the large 3D problem of the bench
        dict(name="grid3d_192", entry="order", shape="grid", a=192, b=192, c=192, options="default", shuffled=False),
        # an unstructured 2D mesh in twenty parts, diagonal stored
        dict(name="mesh_strips_1200k", entry="order", shape="strips", n=1_200_000, regions=20, options="default",
             shuffled=False),
        # a circuit- or network-like matrix with hub rows of thousands of entries
        dict(name="power_law_1m", entry="order", shape="power_law", n=1_000_000, degree=10.0, gamma=2.5,
             options="default", shuffled=False),
        # a solver that holds its matrix on the host
        dict(name="host_100", entry="host", shape="grid", a=100, b=100, c=100, shuffled=False),
        # subdomain blocks of one matrix, ordered once
        dict(name="batch_500", entry="batch", shape="mix", count=500, lo=100, hi=50_000, shuffled=False),
        # the bench's batch, replayed
        dict(name="plan_10000", entry="plan", shape="mix", count=10_000, lo=100, hi=50_000, shuffled=False),
        # a burst of requests of every served size
        dict(name="serve_48", entry="serve", shape="mix", count=48, lo=1_000, hi=4_000_000, shuffled=False),
        # how good an ordering is
        dict(name="bandwidth_192", entry="bandwidth", shape="grid", a=192, b=192, c=192, shuffled=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    entry = rng.choice(("order", "order", "order", "order", "noalloc", "host", "batch", "plan", "serve", "bandwidth"))
    case = dict(entry=entry, shuffled=rng.random() < 0.3)
    if entry in ("batch", "plan", "serve"):
        hi = _log(rng, 2_000, 4_000_000 if entry == "serve" else 50_000)
        count = _log(rng, 8, 48) if entry == "serve" else _log(rng, 30, 10_000 if entry == "plan" else 2_000)
        return dict(case, shape="mix", count=count, lo=rng.randint(100, 1000), hi=hi)
    if entry == "order":
        case["options"] = rng.choice(("default", "default", "default", "l2_window", "components_first", "stored_order"))
    shape = rng.choice(("grid2d", "grid3d", "grid3d", "knn", "strips", "power_law"))
    big = 60_000 if entry == "noalloc" else 7_000_000 if shape == "grid3d" else 1_000_000
    n = _log(rng, 1_000, big)
    if shape == "grid2d":
        a = max(2, int(math.sqrt(n) * rng.uniform(0.7, 1.0)))
        return dict(case, shape="grid", a=a, b=n // a, c=1)
    if shape == "grid3d":
        a = max(2, int(round(n ** (1 / 3) * rng.uniform(0.8, 1.0))))
        b = max(2, int(round(math.sqrt(n / a) * rng.uniform(0.9, 1.0))))
        return dict(case, shape="grid", a=a, b=b, c=max(2, n // (a * b)))
    if shape == "knn":
        return dict(case, shape="knn", n=n, k=rng.choice((2, 3)))
    if shape == "strips":
        return dict(case, shape="strips", n=n, regions=rng.randint(1, 20))
    return dict(case, shape="power_law", n=n, degree=rng.uniform(4, 10), gamma=rng.uniform(2.4, 3.0))


# ---- the patterns, as a symmetric edge list (both directions) over ids that are then permuted ----


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _members(case):
    """(kind, dims) of every graph of a mix: sizes at the middles of equal steps of log n, kinds in turn."""
    lo, hi, count = math.log(case["lo"]), math.log(case["hi"]), case["count"]
    out = []
    for i in range(count):
        n = int(round(math.exp(lo + (hi - lo) * (i + 0.5) / count)))
        if i % 3 == 0:
            r = max(1, int(round(math.sqrt(n))))
            out.append(("grid", (r, max(1, int(round(n / r))), 1)))
        elif i % 3 == 1:
            a = max(1, int(round(n ** (1 / 3))))
            out.append(("grid", (a, a, max(1, int(round(n / (a * a)))))))
        else:
            out.append(("knn", (n, 1, 1)))
    return out


def _spread(values, sizes):
    """values[g] for every vertex of graph g."""
    v = torch.tensor(values, dtype=torch.int64, device="cuda")
    return torch.repeat_interleave(v, torch.tensor(sizes, dtype=torch.int64, device="cuda"))


def _grid_edges(dims, offs):
    """Edges of 2D (c = 1) and 3D stencils, one grid per entry of dims, first vertices at offs."""
    sizes = [a * b * c for a, b, c in dims]
    first = _spread(offs, sizes)
    starts = [0]
    for s in sizes:
        starts.append(starts[-1] + s)
    i = torch.arange(starts[-1], device="cuda") - _spread(starts[:-1], sizes)
    a, b, c = (_spread([d[k] for d in dims], sizes) for k in range(3))
    src, dst = [], []
    for step, at, end in ((1, i % c, c), (c, i // c % b, b), (b * c, i // (b * c), a)):
        m = at + 1 < end
        u = (first + i)[m]
        v = u + (step[m] if torch.is_tensor(step) else step)
        src += [u, v]
        dst += [v, u]
    return torch.cat(src), torch.cat(dst)


def _nearest(x, y, base, side, k):
    """The k nearest points of each point among those of the 3 x 3 cells around it: ids and squared
    distances, -1 where there are fewer. Points come back in cell order: (order, ids, distances)."""
    cx, cy = (x * side).long(), (y * side).long()
    cell = base + cx * side + cy
    cell, order = torch.sort(cell, stable=True)
    x, y, base, side, cx, cy = (t[order] for t in (x, y, base, side, cx, cy))
    count = torch.bincount(cell, minlength=int(cell[-1]) + 2)
    start = torch.cumsum(count, 0) - count
    most, me = int(count.max()), torch.arange(len(x), device="cuda")
    dist = [torch.full_like(x, math.inf) for _ in range(k)]
    ids = [torch.full_like(me, -1) for _ in range(k)]
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            inside = (cx + dx >= 0) & (cx + dx < side) & (cy + dy >= 0) & (cy + dy < side)
            c = (base + (cx + dx) * side + cy + dy).clamp_(0, len(count) - 1)
            left = torch.where(inside, count[c], 0)
            for t in range(most):
                j = (start[c] + t).clamp_(max=len(x) - 1)
                d = torch.where((t < left) & (j != me), (x - x[j]) ** 2 + (y - y[j]) ** 2, math.inf)
                j = torch.where(d < math.inf, j, -1)
                for s in range(k):
                    closer = d < dist[s]
                    dist[s], d = torch.where(closer, d, dist[s]), torch.where(closer, dist[s], d)
                    ids[s], j = torch.where(closer, j, ids[s]), torch.where(closer, ids[s], j)
    return order, torch.stack(ids, 1), torch.stack(dist, 1)


def _knn_edges(sizes, offs, k, gen):
    """Symmetrised k-nearest-neighbour meshes of uniform points, one per entry of sizes."""
    n = sum(sizes)
    x, y = (torch.rand(n, generator=gen, device="cuda") for _ in range(2))
    sides = [max(1, int(math.sqrt(s / 2.5))) for s in sizes]
    cells = [0]
    for s in sides:
        cells.append(cells[-1] + s * s)
    base = _spread(cells[:-1], sizes)
    starts = [0]
    for s in sizes:
        starts.append(starts[-1] + s)
    # points come back sorted by cell, and cells follow their graphs: graph g keeps its places
    _, ids, _ = _nearest(x, y, base, _spread(sides, sizes), k)
    move = _spread([o - s for o, s in zip(offs, starts)], sizes)
    i = torch.arange(n, device="cuda").repeat_interleave(k)
    j = ids.reshape(-1)
    i, j = i[j >= 0], j[j >= 0]
    i, j = i + move[i], j + move[j]
    return torch.cat([i, j]), torch.cat([j, i])


def _spanning_edges(n, u, v, w):
    """Minimum spanning forest (Boruvka) of the weighted edges (u, v): a mask of them."""
    part, keep = torch.arange(n, device="cuda"), torch.zeros(len(u), dtype=torch.bool, device="cuda")
    rank = torch.empty_like(u)
    rank[torch.argsort(w, stable=True)] = torch.arange(len(u), device="cuda")
    edge = torch.argsort(rank)
    while True:
        pu, pv = part[u], part[v]
        out = pu != pv
        if not bool(out.any()):
            return keep
        best = torch.full((n,), len(u), device="cuda")
        best.scatter_reduce_(0, pu[out], rank[out], "amin")
        best.scatter_reduce_(0, pv[out], rank[out], "amin")
        c = torch.nonzero(best < len(u)).squeeze(1)
        e = edge[best[c]]
        keep[e] = True
        to = torch.arange(n, device="cuda")
        to[c] = pu[e] + pv[e] - c
        both = to[to[c]] == c
        to[c[both & (c < to[c])]] = c[both & (c < to[c])]
        while not torch.equal(to, to[to]):
            to = to[to]
        part = to[part]


def _strip_edges(n, regions, gen):
    """Two nearest neighbours and a minimum spanning forest of uniform points in vertical slabs with
    empty strips between them; the diagonal stored."""
    x, y = (torch.rand(n, generator=gen, device="cuda") for _ in range(2))
    cuts = torch.arange(1, regions, device="cuda") / regions
    cuts = cuts + (torch.rand(regions - 1, generator=gen, device="cuda") - 0.5) / regions * 0.8
    region = torch.searchsorted(cuts, x)
    x = x * (1 - 0.002 * (regions - 1)) + 0.002 * region  # a gap of 0.002 between neighbours
    side = torch.full((n,), max(1, int(math.sqrt(n / 2.5))), device="cuda")
    order, ids, dist = _nearest(x, y, torch.zeros_like(side), side, 6)
    region = region[order]
    i, j, w = torch.arange(n, device="cuda").repeat_interleave(6), ids.reshape(-1), dist.reshape(-1)
    near = torch.arange(6, device="cuda").repeat(n) < 2
    ok = j >= 0
    ok[ok.clone()] = region[i[ok]] == region[j[ok]]
    i, j, w, near = i[ok], j[ok], w[ok], near[ok]
    use = near | _spanning_edges(n, i, j, w)
    i, j, own = i[use], j[use], torch.arange(n, device="cuda")
    return torch.cat([i, j, own]), torch.cat([j, i, own])


def _power_law_edges(n, degree, gamma, gen):
    """Edges with both ends drawn with weight (i + 10)^(-1/(gamma - 1)), by the inverse of the weights' integral."""
    e = 1 - 1 / (gamma - 1)
    m = int(round(n * degree / 2))
    low, high = 10 ** e, (n + 10) ** e
    i, j = (((low + (high - low) * torch.rand(m, generator=gen, device="cuda", dtype=torch.float64)) ** (1 / e) - 10)
            .long().clamp_(0, n - 1) for _ in range(2))
    i, j = i[i != j], j[i != j]
    return torch.cat([i, j]), torch.cat([j, i])


def _csr(sizes, src, dst, shuffled, gen):
    """int32 CSR of the edges with every graph's ids permuted among themselves, and the new ids."""
    n = sum(sizes)
    key = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
    if len(sizes) > 1:
        key += _spread(list(range(len(sizes))), sizes)
    new = torch.empty(n, dtype=torch.int64, device="cuda")
    new[torch.argsort(key, stable=True)] = torch.arange(n, device="cuda")
    pair = torch.sort(new[src] * n + new[dst]).values
    del src, dst, key
    pair = torch.unique_consecutive(pair)
    rows = pair // n
    if shuffled:
        at = torch.argsort(rows + torch.rand(len(rows), generator=gen, device="cuda", dtype=torch.float64), stable=True)
        pair, rows = pair[at], rows[at]
    rowptr = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    rowptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return rowptr, (pair - rows * n).to(torch.int32), new


def _pattern(case, seed):
    """(sizes of the graphs, rowptr, colidx, ids of the vertices in the order they were made) of the
    case's pattern, graphs stacked block-diagonally."""
    gen = _generator(seed)
    shape = case["shape"]
    if shape == "grid":
        dims = (case["a"], case["b"], case["c"])
        sizes = [math.prod(dims)]
        src, dst = _grid_edges([dims], [0])
    elif shape == "knn":
        sizes = [case["n"]]
        src, dst = _knn_edges(sizes, [0], case["k"], gen)
    elif shape == "strips":
        sizes = [case["n"]]
        src, dst = _strip_edges(case["n"], case["regions"], gen)
    elif shape == "power_law":
        sizes = [case["n"]]
        src, dst = _power_law_edges(case["n"], case["degree"], case["gamma"], gen)
    else:
        members = _members(case)
        sizes = [math.prod(d) for _, d in members]
        offs = [0]
        for s in sizes:
            offs.append(offs[-1] + s)
        grids = [g for g, (kind, _) in enumerate(members) if kind == "grid"]
        knns = [g for g, (kind, _) in enumerate(members) if kind == "knn"]
        parts = [_grid_edges([members[g][1] for g in grids], [offs[g] for g in grids]),
                 _knn_edges([sizes[g] for g in knns], [offs[g] for g in knns], 3, gen)]
        src, dst = (torch.cat([p[k] for p in parts]) for k in range(2))
    return sizes, *_csr(sizes, src, dst, case["shuffled"], gen)


def _levels(made, seed):
    """An ordering to be judged: front after front in the order the vertices were made (planes of a
    3D grid), each front in random order."""
    n = len(made)
    front = torch.arange(n, device="cuda") // max(1, int(n ** (2 / 3)))
    return made[torch.argsort(front + torch.rand(n, generator=_generator(seed + 1), device="cuda", dtype=torch.float64))]


# ---- the calls ----


class _Handle:
    """A plan or a server that goes with the state that holds it."""

    def __init__(self, made, close):
        status, self.raw = made
        rcm.check(status, "create")
        self._close = close

    def __del__(self):
        torch.cuda.synchronize()
        self._close(self.raw)


def prepare(case, seed):
    sizes, rowptr, colidx, made = _pattern(case, seed)
    n, entry = len(rowptr) - 1, case["entry"]
    state = dict(entry=entry, n=n, rowptr=rowptr, colidx=colidx)
    if entry == "order":
        o = rcm.rcm_options()
        o.l2_persist = 1 if case["options"] == "l2_window" else 0
        o.components_first = 1 if case["options"] == "components_first" else 0
        o.row_order = 1 if case["options"] == "stored_order" else 0
        state["options"] = None if case["options"] == "default" else o
    elif entry == "noalloc":
        state["perm"] = torch.empty(n, dtype=torch.int32, device="cuda")
    elif entry == "host":
        state["rowptr"], state["colidx"] = rowptr.cpu().pin_memory(), colidx.cpu().pin_memory()
        state["perm"] = torch.empty(n, dtype=torch.int32).pin_memory()
    elif entry == "bandwidth":
        state["perm"] = _levels(made, seed).to(torch.int32)
    elif entry == "serve":
        # every request's pattern in pinned host memory, as the serving bench has it
        state["requests"], at = [], 0
        host_rp, host_ci = rowptr.cpu(), colidx.cpu()
        for s in sizes:
            e0, e1 = int(host_rp[at]), int(host_rp[at + s])
            state["requests"].append(((host_rp[at:at + s + 1] - e0).pin_memory(), (host_ci[e0:e1] - at).pin_memory(),
                                      torch.empty(s, dtype=torch.int32).pin_memory()))
            at += s
        del state["rowptr"], state["colidx"]
        state["server"] = _Handle(rcm.rcm_server_create(8 << 30, 256), rcm.rcm_server_destroy)
    else:
        goff = torch.zeros(len(sizes) + 1, dtype=torch.int64)
        goff[1:] = torch.cumsum(torch.tensor(sizes), 0)
        state["goff"] = goff.cuda()
        if entry == "plan":
            state["perm"] = torch.empty(n, dtype=torch.int32, device="cuda")
            state["plan"] = _Handle(rcm.rcm_batch_plan_create(len(sizes), n, len(colidx), state["goff"], rowptr, colidx,
                                                              state["perm"]), rcm.rcm_batch_plan_destroy)
    return state


def run(state):
    entry = state["entry"]
    if entry == "order":
        return rcm.order(state["rowptr"], state["colidx"], state["options"])
    if entry == "batch":
        return rcm.order_batch(state["goff"], state["rowptr"], state["colidx"])
    if entry == "bandwidth":
        return list(rcm.bandwidth_profile(state["rowptr"], state["colidx"], state["perm"]))
    if entry == "plan":
        rcm.check(rcm.rcm_batch_plan_launch(state["plan"].raw), "rcm_batch_plan_launch")
    elif entry == "serve":
        server, tickets = state["server"].raw, []
        for rowptr, colidx, perm in state["requests"]:
            status, ticket = rcm.rcm_submit(server, len(perm), len(colidx), rowptr, colidx, perm)
            rcm.check(status, "rcm_submit")
            tickets.append(ticket)
        for ticket in tickets:
            rcm.check(rcm.rcm_wait(server, ticket), "rcm_wait")
        return [perm for _, _, perm in state["requests"]]
    else:
        call = rcm.rcm_order_noalloc if entry == "noalloc" else rcm.rcm_order_host
        rcm.check(call(state["n"], state["rowptr"], state["colidx"], state["perm"]), entry)
    return state["perm"]


def _size(case):
    """(vertices, stored entries) of the case's pattern; entries of random shapes at their mean."""
    shape = case["shape"]
    if shape == "knn":
        return case["n"], KNN_DEGREE[case["k"]] * case["n"]
    if shape == "strips":
        return case["n"], 3.75 * case["n"]
    if shape == "power_law":
        return case["n"], case["degree"] * case["n"]
    n = nnz = 0
    for kind, (a, b, c) in [("grid", (case["a"], case["b"], case["c"]))] if shape == "grid" else _members(case):
        n += a * b * c
        nnz += KNN_DEGREE[3] * a if kind == "knn" else 2 * (3 * a * b * c - b * c - a * c - a * b)
    return n, nnz


def work(case):
    """The pattern read once and the permutation written once (read, for the bandwidth). All the
    arithmetic is on whole numbers: one operation is one stored entry looked at."""
    n, nnz = _size(case)
    return {"bytes": 4 * (2 * n + 1 + nnz), "flops": nnz}


def exact(case, seed):
    """Bandwidth and profile from their definition. Permutations are whole numbers with no value of
    greater precision: None."""
    if case["entry"] != "bandwidth":
        return None
    _, rowptr, colidx, made = _pattern(case, seed)
    perm = _levels(made, seed)
    n = len(perm)
    pos = torch.empty_like(perm)
    pos[perm] = torch.arange(n, device="cuda")
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), torch.diff(rowptr.long()))
    low = pos.clone().scatter_reduce_(0, rows, pos[colidx.long()], "amin")
    beta = pos - low
    return [int(beta.max()), int(beta.sum())]
