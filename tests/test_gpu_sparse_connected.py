"""Sparse patterns (fewer than 3.2 neighbours a row) that do not fall into parts: trees, cubic and other
sparse random graphs have few, wide levels and belong on the whole grid; the automatic component table must
not take them to one CTA. Patterns of the same density that do fall into parts, or are long and narrow, go
through the probe that gives up. Orderings are compared with the serial oracle, exactly."""
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


def cubic(n, seed):
    """The union of three random perfect matchings: connected with high probability."""
    rng = synth.rng_for(seed)
    p = np.concatenate([rng.permutation(n).reshape(-1, 2) for _ in range(3)])
    return synth.csr_from_edges(n, p[:, 0], p[:, 1])


def beside(parts, seed):
    b = synth.concat(parts)
    return synth.permute(synth.Csr(b.n, b.rowptr, b.colidx), synth.random_permutation(b.n, seed))


def halved(dims, seed):
    """A grid with a vertex in the middle of every edge: 2.4 neighbours a row."""
    g = synth.grid(dims)
    src = np.repeat(np.arange(g.n), np.diff(g.rowptr))
    e = np.stack([src, g.colidx], 1)[src < g.colidx]
    mid = g.n + np.arange(len(e))
    h = synth.csr_from_edges(g.n + len(e), np.concatenate([mid, mid]), e.T.reshape(-1))
    return synth.permute(h, synth.random_permutation(h.n, seed))


def order(rcm, g, **opts):
    o = rcm.rcm_options()
    for k, v in opts.items():
        setattr(o, k, v)
    rp, ci = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (g.rowptr, g.colidx))
    perm, stats = rcm.order(rp, ci, o, with_stats=True)
    return perm.cpu().numpy(), stats


WIDE = {
    "cubic_6k": lambda: cubic(6000, 1),
    "cubic_200k": lambda: cubic(200_000, 2),
    "tree_200k": lambda: synth.random_tree(200_000, 3),
    # a component of 3/4 of the vertices left, and one of a little less, beside small ones
    "most_of_it": lambda: beside([cubic(30_000, 4), cubic(9_000, 5), synth.path(400, seed=6)], 7),
    "giant": lambda: synth.random_graph(100_000, 150_000, seed=8),  # and thousands of small components
}


@pytest.mark.parametrize("first", [0, 1])
@pytest.mark.parametrize("name", list(WIDE))
def test_wide_sparse_graphs_stay_on_the_grid(rcm, name, first):
    g = WIDE[name]()
    got, stats = order(rcm, g, components_first=first)
    assert stats["grid_levels"] > 0
    assert np.array_equal(got, oracle.rcm(g.n, g.rowptr, g.colidx))


NARROW = {
    "path_5k": lambda: synth.path(5000, seed=9),                       # connected: the table has one entry
    "road": lambda: halved((70, 70), 18),                              # connected, and not that thin
    "strips": lambda: synth.knn_mesh(20_000, 2, 10, regions=6),
    "paths": lambda: beside([synth.path(n, seed=n) for n in (33, 32, 31, 34, 65, 64, 63, 66, 130, 2000, 3000, 3001)], 11),
    "just_under": lambda: beside([cubic(20_000, 12), cubic(20_000, 13)], 14),
    # the first start vertex (least degree, least id) lies on a path beside wide parts
    "path_first": lambda: beside([cubic(20_000, 15), synth.path(1500, seed=16)], 17),
}


@pytest.mark.parametrize("opts", [{}, {"fused_sweeps": 1}, {"block_threads": 256}, {"block_threads": 256, "fused_sweeps": -1},
                                  {"narrow_threshold": -1}, {"narrow_threshold": 16}, {"async_sweeps": 1},
                                  {"grid_blocks": 5}, {"expand_mode": 2}, {"components_first": -1}],
                         ids=lambda o: ",".join(f"{k}={v}" for k, v in o.items()) or "default")
@pytest.mark.parametrize("name", list(NARROW))
def test_probe_that_gives_up(rcm, name, opts):
    g = NARROW[name]()
    got, stats = order(rcm, g, **opts)
    want, ref = oracle.rcm(g.n, g.rowptr, g.colidx, with_stats=True)
    assert np.array_equal(got, want)
    # (the oracle counts two sweeps for an isolated vertex, the library none)
    assert stats["components"] == ref["components"]
    assert stats["sweeps"] == ref["sweeps"] - 2 * ref["isolated"]
