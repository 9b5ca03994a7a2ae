"""CTA engines (batches, served requests, components) on graphs whose levels outgrow the shared lists and
table: the sweep goes on in global memory from the first such level, through levels that get narrow again,
and every sweep but the last leaves nothing behind. Orderings equal the serial oracle's, exactly."""
import numpy as np
import pytest

import oracle
from paper_1610_08128_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rcm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1610_08128_gb300 import build, rcm

    build.build()
    rcm.load()
    return rcm


def device(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def necklace(bulbs, width, seed):
    """Wide stars joined by paths: levels of `width` vertices with levels of one between them."""
    src, dst, at = [], [], 0
    for _ in range(bulbs):
        hub, ring, sink = at, np.arange(at + 1, at + 1 + width), at + 1 + width
        src += [np.full(width, hub), ring, np.array([sink, sink + 1])]
        dst += [ring, np.full(width, sink), np.array([sink + 1, sink + 2])]
        at = sink + 2
    g = synth.csr_from_edges(at + 1, np.concatenate(src), np.concatenate(dst))
    return synth.permute(g, synth.random_permutation(g.n, seed))


def beside(parts, seed):
    b = synth.concat(parts)
    return synth.permute(synth.Csr(b.n, b.rowptr, b.colidx), synth.random_permutation(b.n, seed))


GRAPHS = {
    "grid3d_60": lambda: synth.grid((60, 60, 60), seed=1),             # 2,700 vertices in the widest level
    "grid3d_45": lambda: synth.grid((45, 45, 45), seed=2),             # 1,500: at the lists' edge
    "degree_8": lambda: synth.random_graph(20_000, 80_000, seed=3, connected=True),
    "degree_30": lambda: synth.random_graph(6000, 90_000, seed=4, connected=True),
    "power_law": lambda: synth.power_law(20_000, 10.0, 2.5, 5),        # hubs, and small components
    "necklace_2047": lambda: necklace(4, 2047, 6),
    "necklace_2049": lambda: necklace(4, 2049, 7),
    "necklace_700": lambda: necklace(9, 700, 8),
    "two_wide_parts": lambda: beside([synth.random_graph(9000, 40_000, seed=9, connected=True),
                                      synth.grid((50, 50, 50), seed=10), synth.path(700, seed=11)], 12),
}


@pytest.mark.parametrize("threads", [0, 128, 256, 512])
def test_batch(rcm, threads):
    graphs = [make() for make in GRAPHS.values()]
    b = synth.concat(graphs)
    o = rcm.rcm_batch_options()
    o.block_threads = threads
    perm = torch.empty(b.n, dtype=torch.int32, device="cuda")
    rcm.check(rcm.rcm_order_batch_ex(b.G, b.n, device(b.goff), device(b.rowptr), device(b.colidx), perm, o))
    rcm.check(rcm.rcm_stream_status())
    host = perm.cpu().numpy()
    for i, (name, g) in enumerate(zip(GRAPHS, graphs)):
        assert np.array_equal(host[b.goff[i]:b.goff[i + 1]], oracle.rcm(g.n, g.rowptr, g.colidx)), name


@pytest.mark.parametrize("fused", [0, -1, 2])
def test_components(rcm, fused):
    """Wide components beside each other, none of them 3/4 of the vertices."""
    g = beside([make() for make in GRAPHS.values()], 13)
    o = rcm.rcm_options()
    o.fused_sweeps, o.components_first = fused, 1
    got, stats = rcm.order(device(g.rowptr), device(g.colidx), o, with_stats=True)
    want, ref = oracle.rcm(g.n, g.rowptr, g.colidx, with_stats=True)
    assert np.array_equal(got.cpu().numpy(), want)
    assert stats["components"] == ref["components"]
    assert stats["sweeps"] == ref["sweeps"] - 2 * ref["isolated"]  # (the oracle counts two for an isolated vertex)


# What a bitmap takes at most: 1.46M vertices with one CTA on an SM, 0.54M with two (256 threads), 0.08M with
# four (128 threads); a launch whose largest graph is beyond it sizes the others' state smaller.
BEYOND = {
    "one_per_sm": (512, [(1300, 1250), (900, 800), (120, 130)], 0),
    "from_the_sizes": (0, [(1300, 1250), (900, 800), (120, 130)], 0),
    "one_per_sm_256": (256, [(1300, 1250), (900, 800), (120, 130)], 0),
    "two_per_sm": (256, [(800, 700), (700, 690), (60, 70)], 350),
    "four_per_sm": (128, [(300, 280), (280, 270), (60, 70)], 700),
}


@pytest.mark.parametrize("name", list(BEYOND))
def test_graphs_beyond_the_bitmap(rcm, name):
    threads, grids, small = BEYOND[name]
    graphs = [synth.grid_fast(d, seed=i) for i, d in enumerate(grids)] + [synth.path(3, seed=i) for i in range(small)]
    b = synth.concat(graphs)
    o = rcm.rcm_batch_options()
    o.block_threads = threads
    perm = torch.empty(b.n, dtype=torch.int32, device="cuda")
    rcm.check(rcm.rcm_order_batch_ex(b.G, b.n, device(b.goff), device(b.rowptr), device(b.colidx), perm, o))
    rcm.check(rcm.rcm_stream_status())
    host = perm.cpu().numpy()
    for i, g in enumerate(graphs):
        assert np.array_equal(host[b.goff[i]:b.goff[i + 1]], oracle.rcm(g.n, g.rowptr, g.colidx)), i


def with_diagonal(g, rows):
    """The pattern with its first `rows` rows' diagonals stored too."""
    at = np.arange(rows)
    colidx = np.insert(g.colidx, g.rowptr[:rows], at).astype(np.int32)
    return g.rowptr + np.minimum(np.arange(g.n + 1), rows).astype(np.int32), colidx


def test_plan_whose_graphs_grow_beyond_its_bitmap(rcm):
    """A plan made for graphs of 300 vertices, replayed after its buffers were filled with a pattern of the
    same size that has one graph of 20,000 vertices."""
    even = synth.concat([synth.grid((15, 20), seed=i) for i in range(80)])
    grown = synth.concat([synth.grid((100, 200), seed=99)] + [synth.path(50, seed=i) for i in range(80)])
    assert even.n == grown.n and len(grown.colidx) < len(even.colidx)
    rowptr, colidx = with_diagonal(grown, len(even.colidx) - len(grown.colidx))
    fills = [(np.append(even.goff, even.n), even.rowptr, even.colidx), (grown.goff, rowptr, colidx)]
    goff, rp, ci = (device(x) for x in fills[0])
    perm = torch.empty(even.n, dtype=torch.int32, device="cuda")
    st, plan = rcm.rcm_batch_plan_create(len(goff) - 1, even.n, len(ci), goff, rp, ci, perm)
    rcm.check(st, "plan")
    try:
        for at in (0, 1, 0):
            for buf, x in zip((goff, rp, ci), fills[at]):
                buf.copy_(torch.from_numpy(np.ascontiguousarray(x)))
            rcm.check(rcm.rcm_batch_plan_launch(plan))
            rcm.check(rcm.rcm_batch_plan_status(plan))
            host = perm.cpu().numpy()
            for lo, hi in zip(fills[at][0][:-1], fills[at][0][1:]):
                if hi == lo:
                    continue
                r = fills[at][1][lo:hi + 1]
                assert np.array_equal(host[lo:hi], oracle.rcm(int(hi - lo), r - r[0], fills[at][2][r[0]:r[-1]] - lo))
    finally:
        rcm.check(rcm.rcm_batch_plan_destroy(plan))


@pytest.mark.parametrize("rows,length", [(1, 513), (1, 600), (1, 5000), (2, 1000), (12, 520), (40, 900)])
def test_grid_with_dense_rows(rcm, rows, length):
    """Rows of more than 512 entries in a grid, from one in ten thousand entries to one in ten: on both sides
    of the share from which the grid kernel spreads long rows over its warps."""
    g = synth.grid((70, 70, 70))
    rng = synth.rng_for([21, rows, length])
    src = np.repeat(np.arange(g.n), np.diff(g.rowptr))
    hubs = rng.choice(g.n, rows, replace=False)
    ends = np.concatenate([rng.choice(g.n, length, replace=False) for _ in range(rows)])
    h = synth.csr_from_edges(g.n, np.concatenate([src, np.repeat(hubs, length)]), np.concatenate([g.colidx, ends]))
    h = synth.permute(h, synth.random_permutation(h.n, [22, rows]))
    want = oracle.rcm(h.n, h.rowptr, h.colidx)
    for narrow in (0, -1, 700):
        o = rcm.rcm_options()
        o.narrow_threshold = narrow
        got = rcm.order(device(h.rowptr), device(h.colidx), o).cpu().numpy()
        assert np.array_equal(got, want), narrow


@pytest.mark.parametrize("blocks", [2, 8, 0])
@pytest.mark.parametrize("side", [100, 880, 960])
def test_cluster_beside_its_shared_memory(rcm, side, blocks):
    """One cluster on graphs whose bitmap fits beside the full table, beside a small one, and not at all."""
    g = synth.grid_fast((side, side), seed=side)
    o = rcm.rcm_options()
    o.executor, o.cluster, o.grid_blocks = 1, 1, blocks
    got = rcm.order(device(g.rowptr), device(g.colidx), o).cpu().numpy()
    assert np.array_equal(got, oracle.rcm(g.n, g.rowptr, g.colidx))
