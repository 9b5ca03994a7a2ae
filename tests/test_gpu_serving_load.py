"""Served requests on every executor the policy chooses between, under the options' defaults: lone and loaded,
one CTA, clusters of 8 and of 4. Results equal the serial oracle's, exactly."""
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


def serve(rcm, graphs, **opts):
    o = rcm.rcm_server_options()
    for k, v in opts.items():
        setattr(o, k, v)
    st, srv = rcm.rcm_server_create_ex(8 << 30, 256, o)
    rcm.check(st, "create")
    try:
        kept = []
        for g in graphs:
            out = torch.empty(g.n, dtype=torch.int32).pin_memory()
            rp, ci = torch.from_numpy(g.rowptr).pin_memory(), torch.from_numpy(g.colidx).pin_memory()
            s, t = rcm.rcm_submit(srv, g.n, g.nnz, rp, ci, out)
            rcm.check(s, "submit")
            kept.append((rp, ci, out, t))
        for _, _, _, t in kept:
            rcm.check(rcm.rcm_wait(srv, t), "wait")
        return [out.numpy() for _, _, out, _ in kept]
    finally:
        rcm.check(rcm.rcm_server_destroy(srv), "destroy")


def parity(graphs, got):
    want = {}
    for g, p in zip(graphs, got):
        if id(g) not in want:
            want[id(g)] = oracle.rcm(g.n, g.rowptr, g.colidx)
        assert np.array_equal(p, want[id(g)]), g.n


@pytest.fixture(scope="module")
def large():
    return [synth.grid_fast((1030, 1030), seed=1), synth.grid_fast((102, 102, 102), seed=2)]


@pytest.mark.parametrize("dims", [(88, 88, 88), (800, 700), (102, 102, 102)])
def test_lone_request(rcm, dims):
    g = synth.grid_fast(dims, seed=3)
    parity([g], serve(rcm, [g]))


def test_full_server(rcm, large):
    """More requests than count as few: the largest on clusters of 4, the rest on one CTA each."""
    small = [synth.grid((30, 30 + i), seed=i) for i in range(30)] + [synth.power_law(4000, 8.0, 2.5, 5)]
    graphs = small * 4 + large + [synth.grid_fast((88, 88, 88), seed=6)] + large
    parity(graphs, serve(rcm, graphs))


@pytest.mark.parametrize("blocks", [2, 4, 8])
def test_shuffled_rows_on_a_cluster(rcm, blocks):
    graphs = [synth.shuffle_rows(g, [8, i]) for i, g in enumerate(
        [synth.grid((70, 70, 70), seed=7), synth.random_graph(280_000, 1_100_000, 8, connected=True)])]
    parity(graphs, serve(rcm, graphs, cluster_min_vertices=1 << 18, cluster_blocks=blocks))
