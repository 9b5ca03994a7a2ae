"""The sweeps that keep a CTA's traversal state in shared memory, at the sizes where they change path:
bitmap words, passes and list batches of a warp, the list and table capacities (levels beyond them
claim in global memory), the shared frontier cache, rows beyond the padded part, and graphs beyond the
bitmap. Orderings are integers, so parity with the serial oracle is exact equality."""
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


def star_of_stars(arms, leaves, seed):
    """A centre with `arms` neighbours, each with `leaves` leaves: levels of 1, arms, arms * leaves."""
    hub = np.repeat(np.arange(1, arms + 1), leaves)
    leaf = np.arange(arms + 1, arms + 1 + arms * leaves)
    src = np.concatenate([np.zeros(arms, np.int64), hub])
    dst = np.concatenate([np.arange(1, arms + 1), leaf])
    n = 1 + arms + arms * leaves
    return synth.permute(synth.csr_from_edges(n, src, dst), synth.random_permutation(n, seed))


GRAPHS = {
    **{f"path_{n}": (lambda n=n: synth.path(n, seed=n)) for n in (1, 2, 31, 32, 33, 127, 128, 129)},
    **{f"grid_{a}x{b}": (lambda a=a, b=b: synth.grid((a, b), seed=a * b))
       for a, b in ((4, 4), (5, 200), (33, 17), (64, 72), (65, 71))},
    "random_wide": lambda: synth.random_graph(3000, 15000, seed=11, connected=True),       # list overflow
    "random_dense_rows": lambda: synth.random_graph(900, 40000, seed=12, connected=True),  # long rows only
    "random_20k": lambda: synth.random_graph(20000, 60000, seed=13, connected=True),       # beyond the cache
    "arms_40x60": lambda: star_of_stars(40, 60, 14),                                       # 2,400 in a level
    "arms_2100x2": lambda: star_of_stars(2100, 2, 15),                                     # level > cache twice
    "grid3d_40": lambda: synth.grid((40, 40, 40), seed=16),
    "mesh_parts": lambda: synth.knn_mesh(4000, 2, 17),                                     # many components
    "loose": lambda: synth.random_graph(2000, 900, seed=18),                               # isolated vertices
}


def device(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("threads", [0, 32, 128, 512])
def test_small_graphs(rcm, threads):
    for name, make in GRAPHS.items():
        g = make()
        if g.n > 4608:
            continue
        o = rcm.rcm_options()
        o.executor, o.block_threads = 2, threads
        got = rcm.order(device(g.rowptr), device(g.colidx if g.nnz else np.zeros(1, np.int32)), o).cpu().numpy()
        assert np.array_equal(got, oracle.rcm(g.n, g.rowptr, g.colidx)), name


@pytest.mark.parametrize("threads", [0, 128, 256, 512])
@pytest.mark.parametrize("many", [False, True])
def test_batches(rcm, threads, many):
    """All graphs in one batch; with `many`, enough CTAs share an SM that the largest graph exceeds the
    bitmap and is ordered in global memory."""
    graphs = [make() for make in GRAPHS.values()]
    if many:
        graphs += [synth.grid((700, 600), seed=19)] + [synth.path(3, seed=i) for i in range(700)]
    b = synth.concat(graphs)
    o = rcm.rcm_batch_options()
    o.block_threads = threads
    perm = torch.empty(b.n, dtype=torch.int32, device="cuda")
    goff, rp, ci = device(b.goff), device(b.rowptr), device(b.colidx)
    rcm.check(rcm.rcm_order_batch_ex(b.G, b.n, goff, rp, ci, perm, o))
    rcm.check(rcm.rcm_stream_status())
    host = perm.cpu().numpy()
    for i, g in enumerate(graphs):
        assert np.array_equal(host[b.goff[i]:b.goff[i + 1]], oracle.rcm(g.n, g.rowptr, g.colidx)), (i, g.n)


@pytest.mark.parametrize("n", [6000, 40000])
def test_components_of_one_graph(rcm, n):
    """Several components of different widths in one graph, ordered by the component kernel."""
    parts = [synth.grid((70, n // 140), seed=1), synth.random_graph(n // 3, n, seed=2, connected=True),
             star_of_stars(50, n // 200, 3), synth.knn_mesh(n // 6, 2, 4)]
    b = synth.concat(parts)
    g = synth.permute(synth.Csr(b.n, b.rowptr, b.colidx), synth.random_permutation(b.n, 5))
    for first in (0, 1):
        o = rcm.rcm_options()
        o.executor, o.components_first = 1, first
        got = rcm.order(device(g.rowptr), device(g.colidx), o).cpu().numpy()
        assert np.array_equal(got, oracle.rcm(g.n, g.rowptr, g.colidx)), first


@pytest.mark.parametrize("npts", [45000, 50000, 400000])
def test_many_components(rcm, npts):
    """Raw 2-nearest-neighbour meshes: component tables around and well beyond one sort tile."""
    g = synth.knn_mesh(npts, 2, npts)
    got, stats = rcm.order(device(g.rowptr), device(g.colidx), with_stats=True)
    assert stats["components"] > npts // 30
    assert np.array_equal(got.cpu().numpy(), oracle.rcm(g.n, g.rowptr, g.colidx))
